"""harp_grad_blocks on the GPU against the oracle's chain rule, and against invariants at a
configuration's full dimension."""
import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from oracle import harp_oracle as orc
from oracle import harp_params as prm
from paper_2605_29843_b200 import workloads as wl
from harp_testlib import host_rows, promote, to_device

pytestmark = pytest.mark.gpu

DT = {"f32": harp.HARP_F32, "bf16": harp.HARP_BF16}


def _gpu_grad(plan, xh, gh, dtype, accumulate=False, init=None):
    n = xh.shape[0]
    x_d, g_d = to_device(xh, dtype), to_device(gh, dtype)
    n_par = harp.harp_plan_n_params(plan)
    out = torch.full((n_par,), 3.0, dtype=torch.float32, device="cuda") if init is None else init.clone()
    harp.harp_grad_blocks(plan, x_d.data_ptr(), g_d.data_ptr(), n, DT[dtype], out.data_ptr(), accumulate,
                          torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy().astype(np.float64), x_d, g_d


def _flat(grads):
    return np.concatenate([g.ravel() for g in grads])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("radices,perm", [((4,), "identity"), ((2, 2, 2), "random"), ((4, 3, 5), "random"),
                                          ((16, 8, 2), "identity"), ((7, 2), "random"), ((43, 2), "identity")])
def test_grad_blocks_matches_the_oracle(dtype, radices, perm):
    spec = wl.tiny_plan(31, radices, kind="qr", perm=perm, signs=True)
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    rng = np.random.default_rng(32)
    xh = host_rows(rng.standard_normal((29, spec.d)), dtype)
    gh = host_rows(rng.standard_normal((29, spec.d)), dtype)
    got, x_d, g_d = _gpu_grad(plan, xh, gh, dtype)
    want = _flat(orc.grad_blocks(oplan, promote(xh, dtype), promote(gh, dtype)))
    assert got.shape == want.shape == (harp.harp_plan_n_params(plan),)
    # fp32 stage states, fp64 row sums: error relative to the size of the largest entry
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))
    # the inputs are not modified
    assert np.array_equal(x_d.cpu().view(torch.int16 if dtype == "bf16" else torch.int32).numpy(),
                          to_device(xh, dtype).cpu().view(torch.int16 if dtype == "bf16" else torch.int32).numpy())


@pytest.mark.parametrize("radices", [(8, 4, 2), (2, 8), (4, 4, 4), (6, 7), (5, 3, 7), (2, 16), (4, 16, 2), (16, 16)])
def test_rows_spanning_several_slices(radices):
    """More rows than one thread block of the block-owner kernels walks, with a ragged last slice
    and a ragged last batch; radix 8 both at stride one and strided."""
    spec = wl.tiny_plan(35, radices, kind="qr", perm="random", signs=True)
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    rng = np.random.default_rng(36)
    xh = host_rows(rng.standard_normal((71, spec.d)), "f32")
    gh = host_rows(rng.standard_normal((71, spec.d)), "f32")
    got, _, _ = _gpu_grad(plan, xh, gh, "f32")
    want = _flat(orc.grad_blocks(oplan, promote(xh, "f32"), promote(gh, "f32")))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))
    again, _, _ = _gpu_grad(plan, xh, gh, "f32")
    assert np.array_equal(got, again)                       # fixed summation order


@pytest.mark.parametrize("radices", [(4, 2), (2, 2, 2)])
def test_more_rows_of_a_narrow_plan_than_one_grid_holds(radices):
    """The forward kernels take 32 rows per CTA along grid.y (at most 65535): 2097120 rows in one launch."""
    spec = wl.tiny_plan(37, radices, kind="qr", perm="identity", signs=True)
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(38, 2097120 + 45, spec.d, "bf16")
    got, _, _ = _gpu_grad(plan, xh, gh, "bf16")
    want = _flat(orc.grad_blocks(oplan, promote(xh, "bf16"), promote(gh, "bf16")))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))


def test_accumulate_and_row_chunks_add_up():
    spec = wl.tiny_plan(33, (4, 4, 2), kind="qr", perm="random", signs=True)
    plan = harp.plan_from_spec(spec)
    rng = np.random.default_rng(34)
    xh, gh = host_rows(rng.standard_normal((40, 32)), "f32"), host_rows(rng.standard_normal((40, 32)), "f32")
    full, _, _ = _gpu_grad(plan, xh, gh, "f32")
    first, _, _ = _gpu_grad(plan, xh[:15], gh[:15], "f32")
    both, _, _ = _gpu_grad(plan, xh[15:], gh[15:], "f32", accumulate=True,
                           init=torch.from_numpy(first.astype(np.float32)).cuda())
    assert np.max(np.abs(both - full)) <= 1e-5 * np.max(np.abs(full))
    # no rows: the result is zero (or untouched when accumulating)
    n_par = harp.harp_plan_n_params(plan)
    out = torch.full((n_par,), 3.0, dtype=torch.float32, device="cuda")
    harp.harp_grad_blocks(plan, 0, 0, 0, harp.HARP_F32, out.data_ptr())
    assert float(out.abs().max()) == 0.0


def _rows(seed, n, d, dtype):
    rng = np.random.default_rng(seed)
    return host_rows(rng.standard_normal((n, d)), dtype), host_rows(rng.standard_normal((n, d)), dtype)


def test_every_entry_at_full_dimension_cfg2():
    """cfg2's plan (d = 4096, six radix-4 stages, digit-reversal permutation) on 4100 bf16 rows --
    more than one internal row chunk, ragged against every slice size: every entry of every
    stage's gradient against the oracle's chain rule through Algorithm 1."""
    spec = wl.config(2).plans["q"]
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(90, 4100, spec.d, "bf16")
    got, _, _ = _gpu_grad(plan, xh, gh, "bf16")
    want = _flat(orc.grad_blocks(oplan, promote(xh, "bf16"), promote(gh, "bf16")))
    assert got.shape == want.shape
    off = 0
    for t, b in enumerate(spec.radices):                     # per stage, so a quiet stage cannot hide
        n = spec.d * b
        g, w = got[off:off + n], want[off:off + n]
        off += n
        assert np.max(np.abs(g - w)) <= 2e-5 * np.max(np.abs(w)), t


def test_every_entry_at_full_dimension_cfg4():
    """cfg4's plan (d = 14336, radices 16, 16, 8, 7): all entries on 256 rows, and again on a batch
    long enough to cross the internal row chunk."""
    spec = list(wl.config(4).plans.values())[0]
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    for seed, n in ((91, 256), (92, 1203)):
        xh, gh = _rows(seed, n, spec.d, "bf16")
        got, _, _ = _gpu_grad(plan, xh, gh, "bf16")
        want = _flat(orc.grad_blocks(oplan, promote(xh, "bf16"), promote(gh, "bf16")))
        off = 0
        for t, b in enumerate(spec.radices):
            m = spec.d * b
            g, w = got[off:off + m], want[off:off + m]
            off += m
            assert np.max(np.abs(g - w)) <= 2e-5 * np.max(np.abs(w)), (n, t)


def test_euler_identity_at_full_dimension():
    """cfg2's plan (d = 4096, six radix-4 stages, digit-reversal permutation): y is homogeneous of
    degree one in the kernels of every stage, so <K_t, dL/dK_t> = sum(y * G) for each t; y comes
    from harp_apply itself."""
    w = wl.config(2)
    spec = w.plans["q"]
    plan = harp.plan_from_spec(spec)
    n = 512
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((n, spec.d), device="cuda", generator=g)
    G = torch.randn((n, spec.d), device="cuda", generator=g)
    grad = torch.zeros(harp.harp_plan_n_params(plan), dtype=torch.float32, device="cuda")
    harp.harp_grad_blocks(plan, x.data_ptr(), G.data_ptr(), n, harp.HARP_F32, grad.data_ptr())
    y = x.clone()
    harp.apply_(plan, y)
    L = float((y.double() * G.double()).sum())
    off = 0
    for t, b in enumerate(spec.radices):
        k = torch.from_numpy(np.ascontiguousarray(spec.blocks[t], dtype=np.float32)).cuda().flatten()
        got = float((k.double() * grad[off:off + k.numel()].double()).sum())
        off += k.numel()
        assert got == pytest.approx(L, rel=2e-4), t
    assert off == grad.numel()


@pytest.mark.parametrize("cfg", [3, 4, 5])
def test_euler_identity_on_the_wide_plans(cfg):
    """The wide configurations' plans at full dimension (radices 2 and 43; 16, 16, 8, 7; 8, 8, 8, 8, 2),
    bf16 rows: <K_t, dL/dK_t> = L = sum(y * G) for every stage, with y from the fp64 oracle."""
    w = wl.config(cfg)
    spec = list(w.plans.values())[0]
    plan = harp.plan_from_spec(spec)
    oplan = orc.OraclePlan.from_spec(spec)
    rng = np.random.default_rng(80 + cfg)
    n = 96
    xh = host_rows(rng.standard_normal((n, spec.d)), "bf16")
    gh = host_rows(rng.standard_normal((n, spec.d)), "bf16")
    grad, _, _ = _gpu_grad(plan, xh, gh, "bf16")
    L = float(np.sum(orc.forward(oplan, promote(xh, "bf16")) * promote(gh, "bf16")))
    scale = float(np.sqrt(n * spec.d))                      # size of L for independent unit-variance terms
    off = 0
    for t, b in enumerate(spec.radices):
        k = np.asarray(spec.blocks[t], dtype=np.float32).astype(np.float64).ravel()
        got = float(np.dot(k, grad[off:off + k.size]))
        off += k.size
        assert abs(got - L) <= 2e-4 * max(abs(L), scale), (t, b, got, L)
    assert off == grad.size


def test_parameter_gradient_of_a_plan_built_from_theta():
    """One parameter step's worth of Algorithm 3 without the quantizer: plan from theta, L = sum(y * G)
    with y from harp_apply, dL/dK on the GPU, dL/dtheta on the host; compared with central
    differences of the fp64 oracle (theta -> blocks -> forward) on sampled parameters."""
    radices, d = (4, 2, 8), 64
    rng = np.random.default_rng(70)
    theta = [rng.normal(0, 0.3, (d // b, prm.n_params(b))).astype(np.float32) for b in radices]
    perm = rng.permutation(d).astype(np.int32)
    signs = rng.choice(np.array([-1, 1], dtype=np.int8), d)
    plan = harp.harp_plan_create_from_theta(d, radices, perm=perm, signs=signs, theta=theta)
    xh = host_rows(rng.standard_normal((50, d)), "f32")
    gh = host_rows(rng.standard_normal((50, d)), "f32")
    grad, _, _ = _gpu_grad(plan, xh, gh, "f32")

    def loss(th_list):
        blocks = [prm.blocks_from_theta(b, th.astype(np.float64)) for b, th in zip(radices, th_list)]
        op = orc.OraclePlan(d, radices, perm, signs, [np.float32(k) for k in blocks])
        return float(np.sum(orc.forward(op, promote(xh, "f32")) * promote(gh, "f32")))

    off = 0
    for t, b in enumerate(radices):
        n = d * b
        g_theta = harp.harp_grad_theta(b, theta[t], grad[off:off + n].reshape(d // b, b, b))
        off += n
        for c, k in [(0, 0), (d // b - 1, prm.n_params(b) - 1), (3, 0)]:
            h = 1e-3
            tp = [a.astype(np.float64) for a in theta]
            tm = [a.astype(np.float64) for a in theta]
            tp[t][c, k] += h
            tm[t][c, k] -= h
            # the loss is smooth; blocks are rounded to fp32 inside loss(), hence the loose step and bound
            fd = (loss(tp) - loss(tm)) / (2 * h)
            assert abs(g_theta[c, k] - fd) <= 2e-3 * max(1.0, abs(fd)), (t, c, k, g_theta[c, k], fd)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n_rows", [1, 9, 75])
@pytest.mark.parametrize("radices", [(2, 2, 2, 2), (2,) * 9, (2, 2, 2, 2, 4, 4), (3, 4, 4), (4, 4, 3, 4, 4), (8, 16, 7), (16, 16), (8, 8, 2), (7, 4, 8), (4, 8, 3, 16)])
def test_steps_fed_by_asynchronous_copies(dtype, n_rows, radices):
    """Four radix-2 stages a step and two radix-4 ones (at stride one, at multiples of eight, and at a stride of three, whose rows take
    plain loads), stages of radix 7, 8 and 16 on tiles of eight rows (whole and in part, blocks in a row and strided)."""
    spec = wl.tiny_plan(39, radices, kind="qr", perm="identity", signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(40, n_rows, spec.d, dtype)
    got, _, _ = _gpu_grad(plan, xh, gh, dtype)
    want = _flat(orc.grad_blocks(oplan, promote(xh, dtype), promote(gh, dtype)))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("radices", [(2, 2, 2, 2), (4, 4, 4, 4), (8, 8), (16, 7)])
def test_rows_off_sixteen_byte_boundaries(dtype, radices):
    """Rows that start one element behind a 16-byte boundary take the kernels with plain loads; both sums are the same."""
    spec = wl.tiny_plan(41, radices, kind="qr", perm="identity", signs=True)
    plan = harp.plan_from_spec(spec)
    xh, gh = _rows(42, 21, spec.d, dtype)
    got, x_d, g_d = _gpu_grad(plan, xh, gh, dtype)
    for shift_x, shift_g in ((1, 0), (0, 1), (1, 1)):
        bufs = []
        for t, shift in ((x_d, shift_x), (g_d, shift_g)):
            b = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
            b[shift:shift + t.numel()] = t.reshape(-1)
            bufs.append((b, b.data_ptr() + shift * t.element_size()))
        out = torch.zeros(harp.harp_plan_n_params(plan), dtype=torch.float32, device="cuda")
        harp.harp_grad_blocks(plan, bufs[0][1], bufs[1][1], 21, DT[dtype], out.data_ptr(), False, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        # the same fp32 states and fp64 sums in another order: a rounding of the result
        assert np.max(np.abs(out.cpu().numpy() - got)) <= 1e-6 * np.max(np.abs(got))


@pytest.mark.parametrize("n_rows", [445, 900, 2000])
@pytest.mark.parametrize("radices,dtype", [((8, 5, 3), "bf16"), ((8, 5, 3), "f32"), ((3, 3, 8), "bf16"), ((5, 5, 4), "f32"), ((7, 7, 8), "bf16"), ((7, 7, 8), "f32"),
                                           ((8, 5, 5, 5), "bf16"), ((8, 5, 5, 5), "f32"), ((4, 4, 5, 5, 5), "f32"), ((2,), "f32"), ((2, 2), "bf16"), ((2, 3), "bf16")])
def test_permuted_rows_that_are_no_whole_groups_of_pieces(radices, dtype, n_rows):
    """Widths of no multiple of 128 bytes behind a permutation, down to less than a piece of 16; more rows than one group of them a CTA."""
    spec = wl.tiny_plan(43, radices, kind="qr", perm="random", signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(44, n_rows, spec.d, dtype)
    got, _, _ = _gpu_grad(plan, xh, gh, dtype)
    want = _flat(orc.grad_blocks(oplan, promote(xh, dtype), promote(gh, dtype)))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))


def _back_to_back(radices, n_rows, dtype="f32"):
    """Microseconds of a call among others, best of five."""
    spec = wl.tiny_plan(45, radices, kind="qr", perm="identity", signs=True)
    plan = harp.plan_from_spec(spec)
    x = torch.randn((n_rows, spec.d), device="cuda")
    g, out = torch.randn_like(x), torch.zeros(harp.harp_plan_n_params(plan), device="cuda")
    best = float("inf")
    for _ in range(6):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record()
        for _ in range(10):
            harp.harp_grad_blocks(plan, x.data_ptr(), g.data_ptr(), n_rows, DT[dtype], out.data_ptr(), False, torch.cuda.current_stream().cuda_stream)
        ev[1].record()
        torch.cuda.synchronize()
        best = min(best, ev[0].elapsed_time(ev[1]) * 100)
    return best


def test_stages_on_tiles_leave_the_others_their_l1():
    """A stage of radix 39, one thread an element, takes as long behind stages on tiles in shared memory as among its like, but for their
    own time: 1.5 times as long a product (3.0 behind stages that leave it the smallest L1)."""
    mixed, alike = (7, 39, 2, 8), (39, 11, 10)
    per_product = [_back_to_back(r, 1024) / (np.prod(r) * sum(b for b in r if b > 8)) for r in (mixed, alike)]
    assert per_product[0] <= 2.2 * per_product[1], per_product


def _grad_launches(plan, x, g, out):
    before = harp.harp_launch_count()
    harp.harp_grad_blocks(plan, x.data_ptr(), g.data_ptr(), x.shape[0], harp.HARP_F32, out.data_ptr(), False, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return harp.harp_launch_count() - before


def test_states_of_one_thread_per_element_stages_stay_near_l2():
    """32 MB a state of a chunk where a radix has no owner kernel: 10000 rows of d = 1596 in two chunks."""
    spec = wl.tiny_plan(46, (7, 57, 4), kind="qr", perm="identity", signs=True)
    plan = harp.plan_from_spec(spec)
    x = torch.randn((10000, spec.d), device="cuda")
    g = torch.randn_like(x)
    outs = [torch.zeros(harp.harp_plan_n_params(plan), device="cuda") for _ in range(3)]
    one = _grad_launches(plan, x[:5000], g[:5000], outs[0])
    _grad_launches(plan, x[5000:], g[5000:], outs[1])
    assert _grad_launches(plan, x, g, outs[2]) == 2 * one - 1         # the reduction once
    # sums in fp64, rounded to fp32 once in the whole and once in either half
    assert float((outs[0] + outs[1] - outs[2]).abs().max()) <= 1e-6 * float(outs[2].abs().max())


@pytest.mark.parametrize("n_rows", [1, 65, 700])
@pytest.mark.parametrize("radices", [(2, 2, 2), (4, 4, 2), (4, 4, 2, 2, 2), (16, 8, 2), (4, 8, 8, 2)])
def test_a_radix_two_stage_alone(radices, n_rows):
    """Widths of 8 to 512: single blocks up to where fours of them fill a warp (d = 256), fours from there on."""
    spec = wl.tiny_plan(47, radices, kind="qr", perm="identity", signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(48, n_rows, spec.d, "f32")
    got, _, _ = _gpu_grad(plan, xh, gh, "f32")
    want = _flat(orc.grad_blocks(oplan, promote(xh, "f32"), promote(gh, "f32")))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n_rows", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("radices", [(16, 16), (8, 8, 7), (16, 8, 2)])
def test_few_rows_of_wide_stages(dtype, n_rows, radices):
    """One row (radix 16) and three (7 and 8) without tiles of eight, from there on with them."""
    spec = wl.tiny_plan(49, radices, kind="qr", perm="random", signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh, gh = _rows(50, n_rows, spec.d, dtype)
    got, _, _ = _gpu_grad(plan, xh, gh, dtype)
    want = _flat(orc.grad_blocks(oplan, promote(xh, dtype), promote(gh, dtype)))
    assert np.max(np.abs(got - want)) <= 2e-5 * np.max(np.abs(want))


def test_smaller_chunks_where_the_largest_is_not_to_be_had(monkeypatch):
    """Five steps of d = 8192 in fp32: 6000 rows are 1125 MB of states, in two chunks of up to 640 MB, four of 320 and eight of 160; below that
    the call says that it has no memory and writes nothing."""
    spec = wl.tiny_plan(51, (8, 8, 8, 8, 2), kind="qr", perm="identity", signs=True)
    x = torch.randn((6000, spec.d), device="cuda")
    g = torch.randn_like(x)
    n_par = harp.harp_plan_n_params(harp.plan_from_spec(spec))
    want = torch.zeros(n_par, device="cuda")
    launches = _grad_launches(harp.plan_from_spec(spec), x, g, want)
    for limit, chunks in ((1280, 1), (1000, 2), (400, 4), (160, 8)):
        monkeypatch.setenv("HARP_GRAD_SCRATCH_MB", str(limit))
        out = torch.zeros(n_par, device="cuda")
        assert _grad_launches(harp.plan_from_spec(spec), x, g, out) == chunks * (launches - 1) + 1          # one reduction
        # the same fp32 states and fp64 sums in another order: a rounding of the result
        assert float((out - want).abs().max()) <= 1e-6 * float(want.abs().max())
    monkeypatch.setenv("HARP_GRAD_SCRATCH_MB", "100")
    plan, out = harp.plan_from_spec(spec), torch.full((n_par,), 3.0, device="cuda")
    with pytest.raises(harp.HarpError) as e:
        _grad_launches(plan, x, g, out)
    torch.cuda.synchronize()
    assert e.value.status == 9 and bool((out == 3.0).all())
