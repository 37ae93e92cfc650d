"""GPU parity of the matrix path where its cuts lie: tiles of 8 x 16 pixels and runs of the raster,
stages of 64 (fp16), 128 (int8) and 32 (fp32) channels, filter tiles of 32 to 256, pairs of blocks,
reductions split over a cluster, tensor copies against gathered rows."""
import numpy as np
import pytest

import oracle
from paper_2206_10620_b200 import binding, workloads as wl
from _gpu_util import TOL, check_guards, compare, guarded_output, pack, run_gpu

pytestmark = pytest.mark.gpu


def _layer(dtype, n, ci, co, h, w, stride=1, prune=0.5, seed=1, x_dist=None):
    xd = x_dist or {"f32": "upm1", "f16": "relu_normal", "i8": "u01"}[dtype]
    spec = wl.LayerSpec("t", n, ci, co, h, w, stride, dtype, prune, 12, "he", xd, 0.05, True, 0)
    return wl.make_layer(spec, seed=seed)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("shape", [
    (1, 8, 16, 1, 1),         # one pixel
    (1, 16, 31, 1, 9),        # one row, one column past an 8-pixel column, ragged filters
    (3, 17, 33, 16, 8),       # exactly one tile an image; channels of no whole 16 bytes
    (2, 64, 64, 17, 9),       # one row and one column past a tile; one whole stage (fp16)
    (5, 80, 40, 7, 7),        # several small images in a tile
    (2, 144, 129, 15, 29),    # a stage and a piece; one filter past a tile of 128
    (1, 48, 257, 33, 40),     # one filter past the largest tile
    (9, 96, 72, 30, 31),      # runs of the raster over all images
])
def test_edges_of_tiles(dtype, stride, shape):
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, stride, seed=sum(shape))
    pk = pack(d)
    assert pk.plan_info(n, h, w)["matrix_path"] == 1
    compare(d, run_gpu(pk, d.x, d.bias, True))
    compare(d, run_gpu(pk, d.x, None, False), bias=None, relu=False)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("ci", [1, 3, 4, 5, 7, 8])
def test_either_side_of_the_fewest_channels(dtype, stride, ci):
    """fp32 layers of five channels and fp16 / int8 layers of eight are the first on the matrix units."""
    n, co, h, w = 2, 40, 19, 26
    d = _layer(dtype, n, ci, co, h, w, stride, prune=0.2, seed=ci)
    pk = pack(d)
    assert pk.plan_info(n, h, w)["matrix_path"] == int(ci >= (5 if dtype == "f32" else 8))
    compare(d, run_gpu(pk, d.x, d.bias, True))
    compare(d, run_gpu(pk, d.x, None, False, plan=True), bias=None, relu=False)


@pytest.mark.parametrize("dtype", ["f16", "i8"])
@pytest.mark.parametrize("stride,shape", [
    (2, (24, 67, 93, 56, 56)),     # several items of a block, two stages each (int8: one); elements stored one by one
    (2, (24, 131, 40, 41, 57)),    # ... of three stages (two); whole pieces of y
    (2, (30, 17, 37, 64, 50)),     # one short stage
    (2, (6, 503, 256, 28, 28)),    # eight stages (four): fp16 chains that are cut
    (2, (1, 67, 300, 13, 17)),     # one item a block: whole stages
    (1, (3, 67, 93, 45, 77)),      # a raster of 467 entries
    (1, (5, 33, 31, 20, 140)),
    (1, (72, 103, 285, 66, 5)),    # several items of a block, columns of zeros in the raster
])
def test_rows_shifted_in_parts_of_a_stage(dtype, stride, shape):
    """Rows of x that are not whole 16-byte pieces, in tiles too large for the shared memory of whole stages."""
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, stride, seed=ci)
    pk = pack(d)
    assert pk.plan_info(n, h, w)["matrix_path"] == 1
    y = run_gpu(pk, d.x, d.bias, True)
    compare(d, y)
    for _ in range(2):
        assert np.array_equal(run_gpu(pk, d.x, d.bias, True), y)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("shape", [(1, 512, 96, 14, 14), (1, 320, 512, 7, 7), (2, 256, 40, 9, 12)])
def test_reduction_split_over_a_cluster(dtype, shape):
    """Few pixels, many channels: the blocks of a cluster share an item; the result does not depend
    on when they arrive."""
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, prune=0.7, seed=ci)
    pk = pack(d)
    y = run_gpu(pk, d.x, d.bias, True, plan=True)
    compare(d, y)
    for _ in range(3):
        assert np.array_equal(run_gpu(pk, d.x, d.bias, True), y)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("co", [40, 37])
@pytest.mark.parametrize("pool", [0, 2])
def test_fused_operators_behind_tiles_and_splits(dtype, co, pool):
    import torch
    for n, ci, h, w in ((3, 24, 14, 22), (1, 256, 12, 10)):
        d = _layer(dtype, n, ci, co, h, w, seed=co + pool)
        pk = pack(d)
        size = n * h * w * co
        res = (wl.integers(3, "AUX", 1, size, -9999, 9999).astype(np.int32) if dtype == "i8"
               else (wl.normal(3, "AUX", 1, size) * 0.5).astype(np.float32 if dtype == "f32" else np.float16)).reshape(n, h, w, co)
        for scale in ([None, (wl.uniform01(4, "AUX", 2, co) * 2e-3 + 1e-4).astype(np.float32)] if dtype == "i8" else [None]):
            t = torch.uint8 if scale is not None else {"f32": torch.float32, "f16": torch.float16, "i8": torch.int32}[dtype]
            step = 2 if pool else 1
            buf, y = guarded_output((n, h // step, w // step, co), t)
            dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() if a is not None else None for a in (d.x, d.bias, res, scale)]
            p = [0 if a is None else a.data_ptr() for a in dev]
            pk.run_fused(p[0], n, h, w, p[1], y.data_ptr(), relu=True, pool=pool, residual_ptr=p[2], requant_scale_ptr=p[3], zero_point=9)
            pk.sync()
            check_guards(buf)
            ref = oracle.conv_fused(d.x, d.w, d.pid, d.masks, bias=d.bias, relu=True, residual=res, pool=pool, requant_scale=scale, zero_point=9)
            got = y.cpu().numpy()
            if dtype == "i8":
                assert np.array_equal(got.astype(np.int64), ref.astype(np.int64))
            else:
                pre, S = oracle.conv(d.x, d.w, d.pid, d.masks, bias=d.bias, relu=False, with_scale=True)
                bound = TOL[dtype] * np.maximum(np.abs(pre + res), 0.01 * (S + np.abs(res))) + 1e-30
                if pool:
                    bound = bound.reshape(n, h // 2, 2, w // 2, 2, co).max(axis=(2, 4))
                assert (np.abs(got - ref) <= bound).all()


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("co", [1, 2, 65, 129])
def test_residual_of_a_narrow_last_filter_tile(dtype, co):
    """The residual is asked for a tile ahead: rows of a few bytes, the tensor's ends included."""
    import torch
    n, ci, h, w = 2, 16, 9, 17
    d = _layer(dtype, n, ci, co, h, w, seed=co)
    size = n * h * w * co
    res = (wl.integers(5, "AUX", 1, size, -9999, 9999).astype(np.int32) if dtype == "i8"
           else (wl.normal(5, "AUX", 1, size) * 0.5).astype(np.float32 if dtype == "f32" else np.float16)).reshape(n, h, w, co)
    pk = pack(d)
    x, b, r = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (d.x, d.bias, res))
    buf, y = guarded_output((n, h, w, co), {"f32": torch.float32, "f16": torch.float16, "i8": torch.int32}[dtype])
    pk.run_fused(x.data_ptr(), n, h, w, b.data_ptr(), y.data_ptr(), relu=False, residual_ptr=r.data_ptr())
    pk.sync()
    check_guards(buf)
    got, ref = y.cpu().numpy(), oracle.conv_fused(d.x, d.w, d.pid, d.masks, bias=d.bias, relu=False, residual=res)
    if dtype == "i8":
        assert np.array_equal(got.astype(np.int64), ref.astype(np.int64))
    else:
        pre, S = oracle.conv(d.x, d.w, d.pid, d.masks, bias=d.bias, relu=False, with_scale=True)
        assert (np.abs(got - ref) <= TOL[dtype] * np.maximum(np.abs(pre + res), 0.01 * (S + np.abs(res))) + 1e-30).all()


def test_fp32_sums_keep_fp32_precision():
    """Long sums of positive terms, where a truncating accumulator would show: the error stays that of
    a few roundings, and operands keep all of their bits."""
    d = _layer("f32", 1, 512, 64, 16, 16, prune=0.0, seed=5, x_dist="u01")
    d.w = np.abs(d.w)
    y = run_gpu(pack(d), d.x, None, False)
    ref = oracle.conv(d.x, d.w, d.pid, d.masks, bias=None, relu=False)
    assert np.abs(y / ref - 1).max() < 1.5e-6
    d = _layer("f32", 1, 16, 32, 8, 8, prune=0.0, seed=6)
    d.x[:] = 0
    d.x[0, 4, 4, 3] = np.float32(3.4e38)                 # above the largest bf16, below the largest fp32
    d.w[:] = 0
    d.w[7, 3] = np.float32(2.0 ** -100)
    ref = oracle.conv(d.x, d.w, d.pid, d.masks, bias=None, relu=False)
    np.testing.assert_allclose(run_gpu(pack(d), d.x, None, False), ref, rtol=1e-6, atol=0)


@pytest.mark.parametrize("ci", [512, 1024, 4096])
def test_fp16_sums_of_many_channels(ci):
    """Matrix instructions truncate when they add: a step loses less than a unit of the accumulator's last
    place, 2^-23 of the sum so far; half of one on the average, and of a sum that on the average is half there, so
    2^-25 a step of the whole where all terms are positive.  No chain is longer than 288 steps."""
    d = _layer("f16", 2, ci, 64, 16, 16, prune=0.0, seed=ci)
    d.w = np.abs(d.w)
    pk = pack(d)
    assert pk.plan_info(74, 16, 16)["matrix_splits"] == 1
    y = run_gpu(pk, np.tile(d.x, (37, 1, 1, 1)), None, False)
    assert np.array_equal(y[:2], y[-2:])
    ref = oracle.conv(d.x, d.w, d.pid, d.masks, bias=None, relu=False)
    steps = min(9 * (ci // 16), 288)
    assert (np.abs(y[:2] - ref) <= (2.0 ** -11 + steps * 2.0 ** -23) * ref + 2.0 ** -25).all()
    # (the mean of 2^15 roundings to fp16 is within 2^-11 / 2^7 of none)
    assert -steps * 2.0 ** -25 - 2.0 ** -18 <= (y[:2] / ref - 1).mean() <= 2.0 ** -18


@pytest.mark.parametrize("n,ci,co,hw,stride", [
    (74, 600, 64, 16, 1),         # two accumulators, cut every 4 stages, a short last part
    (74, 600, 64, 32, 2),
    (74, 640, 256, 16, 1),        # one accumulator, cut every 8 stages, pairs of blocks
    (40, 640, 256, 20, 1),        # two tiles a block
    (10, 4096, 64, 16, 1),        # split over a cluster and cut
])
def test_fp16_chains_that_are_cut(n, ci, co, hw, stride):
    d = _layer("f16", 1, ci, co, hw, hw, stride, prune=0.4, seed=ci + co)
    x = np.tile(d.x, (n, 1, 1, 1))
    y = run_gpu(pack(d), x, d.bias, True)
    assert (y == y[:1]).all()
    compare(d, y[:1])


@pytest.mark.parametrize("m,k,co", [(20000, 4700, 256), (20000, 4616, 40), (300, 6000, 100)])
def test_fp16_products_whose_chains_are_cut(m, k, co):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", 100, k, co, 16, 16, 0.7, 0.7, "f16"), seed=k)
    g = binding.BlockGemm(k, co, 16, 16, "f16", d.w, d.row_keep, d.col_keep)
    x, b = torch.from_numpy(d.x).cuda().repeat(m // 100, 1), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output((m, co), torch.float16)
    g.run(x.data_ptr(), m, b.data_ptr(), True, y.data_ptr())
    g.sync()
    check_guards(buf)
    got = y.cpu().numpy().reshape(-1, 100, co)
    assert (got == got[:1]).all()
    ref, S = oracle.block_gemm(d.x, d.w, d.row_keep, d.col_keep, 16, 16, bias=d.bias, relu=True, with_scale=True)
    assert (np.abs(got[0].astype(np.float64) - ref) <= TOL["f16"] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25).all()


def _sum_of_kept(x, w, keep, stride):
    """Sums over the kept weights alone, zeros around the image; fp64, infinities as they come."""
    n, h, wd, _ = x.shape
    ho, wo = (h - 1) // stride + 1, (wd - 1) // stride + 1
    xp = np.zeros((n, h + 2, wd + 2, x.shape[3]))
    xp[:, 1:-1, 1:-1] = x
    y = np.zeros((n, ho, wo, w.shape[0]))
    with np.errstate(invalid="ignore"):
        for t in range(9):
            xt = xp[:, t // 3:t // 3 + stride * (ho - 1) + 1:stride, t % 3:t % 3 + stride * (wo - 1) + 1:stride]
            for oc in range(w.shape[0]):
                k = np.flatnonzero(keep[oc, :, t])
                y[..., oc] += (xt[..., k] * w[oc, k, t].astype(np.float64)).sum(axis=-1)
    return y


def _same_with_infinities(got, ref, S, dtype):
    got = got.astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    far = np.isinf(ref)
    assert np.array_equal(got[far], ref[far])
    ok = np.isfinite(ref)
    assert ok.any() and far.any()
    assert (np.abs(got[ok] - ref[ok]) <= TOL[dtype] * np.maximum(np.abs(ref[ok]), 0.01 * S[ok]) + 2.0 ** -25).all()


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("shape", [
    (2, 3, 32, 18, 11),       # the command-stream kernel
    (2, 5, 32, 18, 11),       # (fp32: the fewest channels of the matrix path)
    (2, 16, 32, 18, 11),
    (1, 40, 37, 9, 17),       # gathered rows, staged stores
    (1, 256, 40, 10, 12),     # split over a cluster
    (9, 72, 96, 30, 31),      # runs of the raster
])
def test_infinities_reach_kept_weights_alone(dtype, stride, shape):
    """A pruned weight contributes nothing, whatever it would be multiplied by; a kept one an infinity or a
    NaN, as IEEE arithmetic has it.  Infinite weights, and kept zeros, likewise."""
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, stride, prune=0.6, seed=sum(shape))
    taps = np.array([[(int(m) >> t) & 1 for t in range(9)] for m in d.masks], bool)
    keep = (d.pid.reshape(co, ci)[..., None] >= 0) & taps[d.pid.reshape(co, ci)]
    rng = np.random.default_rng(ci)
    for v in (np.inf, -np.inf, np.nan, np.inf):
        d.x[rng.integers(n), rng.integers(h), rng.integers(w), rng.integers(ci)] = v
    wt = d.w.reshape(co, ci, 9)
    wt[0, 0] = 0                                          # kept zeros
    d.x[0, h // 2, w // 2, 0] = np.inf
    o, c = np.argwhere(keep.any(-1))[-1]
    wt[o, c] = np.inf
    S = _sum_of_kept(np.abs(np.where(np.isfinite(d.x), d.x, 0)), np.abs(np.where(np.isfinite(wt), wt, 0)), keep, stride)
    y = run_gpu(pack(d), d.x, None, False)
    _same_with_infinities(y, _sum_of_kept(d.x, wt, keep, stride), S, dtype)


@pytest.mark.parametrize("dtype,n,ci,co,hw", [
    ("f16", 16, 128, 256, 28),    # two tiles a block
    ("f16", 48, 256, 256, 28),    # pairs of blocks, several items each
    ("f32", 48, 128, 256, 28),    # pairs, several items
    ("f16", 74, 600, 64, 16),     # chains that are cut
    ("f16", 10, 4096, 64, 16),    # split and cut
])
def test_infinities_in_every_item_of_a_block(dtype, n, ci, co, hw):
    """The same image over and over: what is computed anew does not depend on the place."""
    d = _layer(dtype, 1, ci, co, hw, hw, prune=0.6, seed=ci)
    taps = np.array([[(int(m) >> t) & 1 for t in range(9)] for m in d.masks], bool)
    keep = (d.pid.reshape(co, ci)[..., None] >= 0) & taps[d.pid.reshape(co, ci)]
    d.x[0, 3, 4, 5], d.x[0, hw - 1, hw - 1, ci - 1], d.x[0, 9, 0, 1] = np.inf, -np.inf, np.nan
    y = run_gpu(pack(d), np.tile(d.x, (n, 1, 1, 1)), None, False)
    assert np.array_equal(y, np.broadcast_to(y[:1], y.shape), equal_nan=True)
    w = d.w.reshape(co, ci, 9)
    S = _sum_of_kept(np.abs(np.where(np.isfinite(d.x), d.x, 0)), np.abs(w), keep, 1)
    _same_with_infinities(y[:1], _sum_of_kept(d.x, w, keep, 1), S, dtype)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("ci", [24, 256])
def test_infinities_under_a_pool_and_a_residual(dtype, ci):
    import torch
    n, co, h, w = 1, 40, 12, 10
    d = _layer(dtype, n, ci, co, h, w, prune=0.6, seed=ci)
    taps = np.array([[(int(m) >> t) & 1 for t in range(9)] for m in d.masks], bool)
    keep = (d.pid.reshape(co, ci)[..., None] >= 0) & taps[d.pid.reshape(co, ci)]
    d.x[0, 3, 4, 5], d.x[0, 8, 8, 1] = np.inf, -np.inf
    res = (wl.normal(3, "AUX", 1, n * h * w * co) * 0.5).astype(d.x.dtype).reshape(n, h, w, co)
    v = _sum_of_kept(d.x, d.w.reshape(co, ci, 9), keep, 1)
    S = _sum_of_kept(np.abs(np.where(np.isfinite(d.x), d.x, 0)), np.abs(d.w.reshape(co, ci, 9)), keep, 1)
    for pool, r in ((0, res), (2, None), (2, res)):
        ref, s = v + (0 if r is None else r.astype(np.float64)), S + (0 if r is None else np.abs(r))
        if pool:
            ref, s = (a.reshape(n, h // 2, 2, w // 2, 2, co).max(axis=(2, 4)) for a in (ref, s))
        buf, y = guarded_output(ref.shape, torch.float32 if dtype == "f32" else torch.float16)
        x, rt = torch.from_numpy(d.x).cuda(), torch.from_numpy(res).cuda()
        pk = pack(d)
        pk.run_fused(x.data_ptr(), n, h, w, 0, y.data_ptr(), relu=False, pool=pool, residual_ptr=0 if r is None else rt.data_ptr())
        pk.sync()
        check_guards(buf)
        _same_with_infinities(y.cpu().numpy(), ref, s, dtype)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("m,k,co", [(300, 72, 80), (33, 1000, 50)])
def test_infinities_of_the_block_pruned_product(dtype, m, k, co):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", m, k, co, 16, 16, 0.5, 0.5, dtype), seed=m + k)
    keep = np.zeros((co, k), bool)
    for o in range(co):
        for c in range(k):
            keep[o, c] = d.row_keep[o // 16, c // 16, o % 16] and d.col_keep[o // 16, c // 16, c % 16]
    d.x[1, 3], d.x[2, 5], d.x[m - 1, k - 1], d.x[0, 20] = np.inf, np.nan, -np.inf, np.inf
    g = binding.BlockGemm(k, co, 16, 16, dtype, d.w, d.row_keep, d.col_keep)
    x = torch.from_numpy(d.x).cuda()
    buf, y = guarded_output((m, co), torch.float32 if dtype == "f32" else torch.float16)
    g.run(x.data_ptr(), m, 0, False, y.data_ptr())
    g.sync()
    check_guards(buf)
    ref, S = np.zeros((m, co)), np.zeros((m, co))
    with np.errstate(invalid="ignore"):
        for o in range(co):
            c = np.flatnonzero(keep[o])
            p = d.x[:, c].astype(np.float64) * d.w.reshape(co, k)[o, c].astype(np.float64)
            ref[:, o], S[:, o] = p.sum(axis=1), np.abs(np.where(np.isfinite(p), p, 0)).sum(axis=1)
    _same_with_infinities(y.cpu().numpy(), ref, S, dtype)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("m", [1, 127, 129, 1000])
@pytest.mark.parametrize("k,co", [(16, 32), (33, 31), (200, 264)])
def test_block_pruned_product(dtype, m, k, co):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", m, k, co, 16, 16, 0.5, 0.5, dtype), seed=m + k)
    g = binding.BlockGemm(k, co, 16, 16, dtype, d.w, d.row_keep, d.col_keep)
    ref, S = oracle.block_gemm(d.x, d.w, d.row_keep, d.col_keep, 16, 16, bias=d.bias, relu=True, with_scale=True)
    bound = TOL[dtype] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25
    t = torch.float32 if dtype == "f32" else torch.float16
    for shift in (0, 1):                                 # tensors that start on an element, not on 16 bytes
        x = torch.zeros(m * k + shift, dtype=t, device="cuda")
        x[shift:] = torch.from_numpy(d.x).cuda().reshape(-1)
        buf, y = guarded_output((m, co), t)
        b = torch.from_numpy(d.bias).cuda()
        g.run(x.data_ptr() + shift * x.element_size(), m, b.data_ptr(), True, y.data_ptr())
        torch.cuda.synchronize()
        check_guards(buf)
        assert (np.abs(y.cpu().numpy().astype(np.float64) - ref) <= bound).all()


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("shape", [
    (1, 16, 32, 8, 8),        # one stage, one item
    (40, 64, 64, 40, 40),     # several items a block (fp32: pairs of blocks)
    (32, 256, 256, 28, 28),   # pairs of blocks, several stages
    (2, 48, 200, 60, 60),     # several filter tiles
    (1, 512, 96, 14, 14),     # split over a cluster
])
def test_a_wait_that_runs_out_is_reported(dtype, shape):
    """Stages told to wait for an arrival that never comes: every wait ends at its (shortened) limit, the
    kernel ends by itself and stays inside its tensors, the timeout is reported once, and the next run is
    as the one before."""
    import torch
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, seed=sum(shape))
    pk = pack(d)
    pk.plan(n, h, w, wait_limit_ms=20)
    assert pk.plan_info(n, h, w)["matrix_path"] == 1
    before = run_gpu(pk, d.x, d.bias, True)
    pk.test_expect_arrivals(1)
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output((n, h, w, co), {"f32": torch.float32, "f16": torch.float16, "i8": torch.int32}[dtype])
    pk.run(x.data_ptr(), n, h, w, b.data_ptr(), True, y.data_ptr())            # only enqueues: OK
    with pytest.raises(binding.PatconvError) as e:
        pk.sync()
    assert e.value.status == 7
    check_guards(buf)
    pk.sync()                                                                  # reported once
    pk.test_expect_arrivals(0)
    assert np.array_equal(run_gpu(pk, d.x, d.bias, True), before)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("m,k,co", [(5, 16, 32), (40000, 200, 264), (96, 1000, 500)])
def test_a_wait_of_the_block_pruned_product_that_runs_out_is_reported(dtype, m, k, co):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", m, k, co, 16, 16, 0.5, 0.5, dtype), seed=m + k)
    g = binding.BlockGemm(k, co, 16, 16, dtype, d.w, d.row_keep, d.col_keep)
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output((m, co), torch.float32 if dtype == "f32" else torch.float16)
    run = lambda: g.run(x.data_ptr(), m, b.data_ptr(), True, y.data_ptr())
    g.test_expect_arrivals(1)
    run()
    with pytest.raises(binding.PatconvError) as e:
        g.sync()
    assert e.value.status == 7
    check_guards(buf)
    g.sync()
    g.test_expect_arrivals(0)
    y.fill_(777.0)
    run()
    g.sync()
    rows = min(m, 512)
    ref, S = oracle.block_gemm(d.x[-rows:], d.w, d.row_keep, d.col_keep, 16, 16, bias=d.bias, relu=True, with_scale=True)
    bound = TOL[dtype] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25
    assert (np.abs(y.cpu().numpy()[-rows:].astype(np.float64) - ref) <= bound).all()


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("shape", [(1, 6, 1, 1), (2, 2, 13, 5), (1, 20, 40, 33), (40, 64, 17, 30), (3, 7, 2, 9)])
def test_depthwise_pieces_of_rows(dtype, stride, shape):
    import torch
    n, c, h, w = shape
    d = wl.make_depthwise(wl.DepthwiseSpec("t", n, c, h, w, stride, dtype, 0.2, 12), seed=c)
    dw = binding.Depthwise(c, stride, dtype, d.masks, d.w, d.pid)
    t = torch.float32 if dtype == "f32" else torch.float16
    ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
    buf, y = guarded_output((n, ho, wo, c), t)
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    dw.run(x.data_ptr(), n, h, w, b.data_ptr(), True, y.data_ptr())
    torch.cuda.synchronize()
    check_guards(buf)
    ref, S = oracle.depthwise(d.x, d.w, d.pid, d.masks, bias=d.bias, relu=True, stride=stride, with_scale=True)
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref)
    assert (err <= TOL[dtype] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25).all()


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("k,co,block", [(520, 1100, 1), (600, 1000, 32)])     # keep flags beyond 1 MB; several pieces of weights
def test_weights_uploaded_in_pieces(dtype, k, co, block):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", 9, k, co, block, block, 0.5, 0.5, dtype), seed=block)
    g = binding.BlockGemm(k, co, block, block, dtype, d.w, d.row_keep, d.col_keep)
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output((9, co), torch.float32 if dtype == "f32" else torch.float16)
    g.run(x.data_ptr(), 9, b.data_ptr(), True, y.data_ptr())
    g.sync()
    check_guards(buf)
    ref, S = oracle.block_gemm(d.x, d.w, d.row_keep, d.col_keep, block, block, bias=d.bias, relu=True, with_scale=True)
    bound = TOL[dtype] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25
    assert (np.abs(y.cpu().numpy().astype(np.float64) - ref) <= bound).all()


def test_calls_report_errors():
    pk = pack(_layer("f32", 1, 16, 32, 8, 8))
    with pytest.raises(binding.PatconvError) as e:
        pk.run(0, 1, 8, 8, 0, True, 16)
    assert e.value.status == 1
    with pytest.raises(TypeError):
        binding._calls.conv(pk._h.value, 0)
    pk.close()
    with pytest.raises(binding.PatconvError) as e:
        pk.run(16, 1, 8, 8, None, True, 4096)
    assert e.value.status == 1


@pytest.mark.parametrize("co", [17, 32, 40, 96])
@pytest.mark.parametrize("ci,stride", [(24, 1), (50, 1), (160, 1), (160, 2)])
def test_fp32_tiles_of_few_filters(co, ci, stride):
    """Items of one to many stages, several to a block, in chunks that go round the epilogue's warps or stay."""
    n, h = (90, 23) if stride == 1 else (40, 61)
    d = _layer("f32", 1, ci, co, h, h, stride, prune=0.4, seed=co + ci)
    y = run_gpu(pack(d), np.tile(d.x, (n, 1, 1, 1)), d.bias, True)
    assert (y == y[:1]).all()
    compare(d, y[:1])


@pytest.mark.parametrize("m,k,co", [(60000, 40, 32), (60000, 200, 20), (40000, 352, 96)])
def test_fp32_products_of_few_filters(m, k, co):
    d = wl.make_block_gemm(wl.GemmSpec("t", 600, k, co, 16, 16, 0.5, 0.5, "f32"), seed=k)
    import torch
    g = binding.BlockGemm(k, co, 16, 16, "f32", d.w, d.row_keep, d.col_keep)
    x, b = torch.from_numpy(np.tile(d.x, (m // 600 + 1, 1))[:m]).cuda(), torch.from_numpy(d.bias).cuda()
    y = torch.empty((m, co), device="cuda")
    g.run(x.data_ptr(), m, b.data_ptr(), True, y.data_ptr())
    g.sync()
    y = y.cpu().numpy()
    assert all((y[i:i + 600] == y[:len(y[i:i + 600])]).all() for i in range(600, m, 600))
    ref, S = oracle.block_gemm(d.x, d.w, d.row_keep, d.col_keep, 16, 16, bias=d.bias, relu=True, with_scale=True)
    assert (np.abs(y[:600] - ref) <= TOL["f32"] * np.maximum(np.abs(ref), 0.01 * S) + 1e-30).all()


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("ci", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("n,h,w,co,stride", [
    (1, 5, 3, 16, 1),             # one pixel a thread, one group of filters
    (2, 40, 61, 33, 1),           # two; three groups, filters that are not whole pieces
    (3, 90, 131, 70, 2),          # more than 64 filters
    (4, 111, 113, 64, 1),         # four
])
def test_few_channels(dtype, ci, n, h, w, co, stride):
    if dtype == "f32" and ci > 4:
        pytest.skip("on the matrix units")
    # (no zeros in x: where all of a window is zero the result is the bias, and half a spacing of fp16's subnormals,
    # 2^-25, is more than 2e-3 of a bias below 1.5e-5)
    d = _layer(dtype, n, ci, co, h, w, stride, prune=0.3, seed=ci + co, x_dist="u01" if dtype == "i8" else "upm1")
    compare(d, run_gpu(pack(d), d.x, d.bias, True))


@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_few_channels_infinities_under_pruned_weights(dtype):
    """As on the command stream, which goes through the kept weights alone."""
    d = _layer(dtype, 1, 3, 32, 20, 30, prune=0.6, seed=3)
    d.x[0, 7, 11, 1] = np.inf
    d.x[0, 15, 20, 0] = np.nan
    stream = pack(d)
    stream.plan(1, 20, 30, splits=1)
    y, ref = run_gpu(pack(d), d.x, d.bias, False).astype(np.float64), run_gpu(stream, d.x, d.bias, False).astype(np.float64)
    fine = np.isfinite(ref)
    assert np.array_equal(np.isfinite(y), fine) and 0 < (~fine).sum() < 2 * 9 * 32
    assert np.array_equal(y[~fine], ref[~fine], equal_nan=True)
    assert (np.abs(y[fine] - ref[fine]) <= 2 * TOL[dtype] * np.maximum(np.abs(ref[fine]), 0.01)).all()


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("co", [32, 37])          # whole pieces of y; elements one by one
def test_few_channels_relu_of_a_nan(dtype, co):
    """The same, with and without other operators behind it, as on the command stream: 0."""
    d = _layer(dtype, 1, 3, co, 20, 30, prune=0.6, seed=4)
    d.x[0, 7, 11, 1] = np.inf                     # (infinite sums of both signs)
    d.x[0, 7, 12, 1] = -np.inf                    # (and sums of both: NaN)
    d.x[0, 15, 20, 0] = np.nan
    few, stream = pack(d), pack(d)
    stream.plan(1, 20, 30, splits=1)
    raw, ref = run_gpu(stream, d.x, d.bias, False), run_gpu(stream, d.x, d.bias, True).astype(np.float64)
    y = run_gpu(few, d.x, d.bias, True).astype(np.float64)
    assert np.isnan(raw).sum() > 20 and not np.isnan(ref).any() and (y[np.isnan(raw)] == 0).all()
    assert np.array_equal(np.isinf(y), np.isinf(ref)) and np.isinf(y).any()
    fine = np.isfinite(ref)
    assert (np.abs(y[fine] - ref[fine]) <= 2 * TOL[dtype] * np.maximum(np.abs(ref[fine]), 0.01)).all()


@pytest.mark.parametrize("ci,co", [(3, 32), (3, 37), (64, 32)])       # dense on the FP32 pipe, whole pieces and not; matrix units
def test_int32_results_wrap(ci, co):
    d = _layer("i8", 1, ci, co, 9, 11, prune=0.3, seed=ci)
    bias = np.where(np.arange(co) % 2, 2 ** 31 - 1, -2 ** 31).astype(np.int32)
    ref = oracle.conv(d.x, d.w, d.pid, d.masks, bias=None, relu=False).astype(np.int64) + bias
    wrapped = (ref + 2 ** 31) % 2 ** 32 - 2 ** 31
    assert (wrapped != ref).any()
    assert np.array_equal(run_gpu(pack(d), d.x, bias, False).astype(np.int64), wrapped)
    assert np.array_equal(run_gpu(pack(d), d.x, bias, True).astype(np.int64), np.maximum(wrapped, 0))


@pytest.mark.parametrize("dtype,ci", [("f32", 4), ("f16", 7), ("i8", 7)])
@pytest.mark.parametrize("co,prune,few", [(96, 0.9, 0), (33, 0.9, None), (64, 0.0, None)])
def test_few_channels_on_either_kernel(dtype, ci, co, prune, few):
    """A large image of which little is left runs on the command stream, with the results of the dense kernel."""
    n, h, w = 1, 224, 210
    d = _layer(dtype, n, ci, co, h, w, prune=prune, seed=co, x_dist="u01" if dtype == "i8" else "upm1")
    pk = pack(d)
    assert few is None or pk.plan_info(n, h, w)["few_channel_path"] == few
    compare(d, run_gpu(pk, d.x, d.bias, True))
    dense = pack(d)
    compare(d, _run_static(dense, d))


def _run_static(pk, d):
    import torch
    s = d.spec
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output((s.n, s.h, s.w, s.c_out), {"f32": torch.float32, "f16": torch.float16, "i8": torch.int32}[s.dtype])
    pk.run_static_scratch(x.data_ptr(), s.n, s.h, s.w, b.data_ptr(), True, y.data_ptr(), 1)
    pk.sync()
    check_guards(buf)
    return y.cpu().numpy()


@pytest.mark.parametrize("dtype,stride,shape", [
    ("f16", 2, (24, 67, 93, 56, 56)),      # rows shifted into place, several stages a block
    ("i8", 2, (24, 67, 93, 56, 56)),
    ("f32", 1, (16, 264, 200, 28, 28)),    # pairs of blocks whose weights stream
    ("f16", 1, (32, 1024, 256, 14, 14)),   # chains that are cut
])
def test_roles_end_where_a_wait_gives_up(dtype, stride, shape):
    """However many stages are left, a launch that gave up ends soon: nobody goes on filling buffers for the others."""
    import time
    import torch
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, stride, seed=ci)
    pk = pack(d)
    pk.plan(n, h, w, wait_limit_ms=20)
    before = run_gpu(pk, d.x, d.bias, True)
    pk.test_expect_arrivals(1)
    x, b = torch.from_numpy(d.x).cuda(), torch.from_numpy(d.bias).cuda()
    buf, y = guarded_output(before.shape, {"f32": torch.float32, "f16": torch.float16, "i8": torch.int32}[dtype])
    torch.cuda.synchronize()
    t0 = time.monotonic()
    pk.run(x.data_ptr(), n, h, w, b.data_ptr(), True, y.data_ptr())
    with pytest.raises(binding.PatconvError) as e:
        pk.sync()
    assert e.value.status == 7 and time.monotonic() - t0 < 1.0
    check_guards(buf)
    pk.test_expect_arrivals(0)
    assert np.array_equal(run_gpu(pk, d.x, d.bias, True), before)
