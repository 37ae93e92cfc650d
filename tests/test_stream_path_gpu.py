"""GPU parity of the kernels that execute a command stream: what a handle runs whose caller names one of
their tuning parameters (the defaults run on the matrix units, see test_matrix_path_gpu.py)."""
import itertools

import numpy as np
import pytest

import oracle
from paper_2206_10620_b200 import binding, workloads as wl
from _gpu_util import TOL, check_guards, compare, guarded_output, pack, run_gpu
from test_fused_gpu import _residual, compare_fused, run_fused

pytestmark = pytest.mark.gpu

ALL_MASKS = np.array([sum(1 << t for t in c) for c in itertools.combinations(range(9), 4)], np.uint16)


def _layer(dtype, n, ci, co, h, w, stride=1, prune=0.5, lib=12, seed=1):
    xd = {"f32": "upm1", "f16": "relu_normal", "i8": "u01"}[dtype]
    return wl.make_layer(wl.LayerSpec("t", n, ci, co, h, w, stride, dtype, prune, lib, "he", xd, 0.05, True, 0), seed=seed)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("shape,lib", [
    ((1, 8, 16, 1, 1), 4),         # one pixel
    ((1, 16, 31, 1, 9), 8),        # one row; ragged filters
    ((3, 17, 33, 16, 8), 12),      # channels of no whole 16 bytes
    ((2, 64, 64, 17, 9), 4),       # one row and one column past the tiling of a warp
    ((5, 80, 40, 7, 7), 8),        # several small images
    ((2, 144, 129, 15, 29), 12),   # several blocks of filters, a last one of one filter
    ((9, 96, 72, 30, 31), 12),     # many items
    ((1, 320, 48, 10, 10), 8),     # int8: totals beyond 24 bits
])
def test_unsplit_and_split(dtype, stride, shape, lib):
    n, ci, co, h, w = shape
    d = _layer(dtype, n, ci, co, h, w, stride, lib=lib, seed=sum(shape))
    pk = pack(d)
    for splits in (1, 3):
        pk.plan(n, h, w, splits=splits, reduce_mode=1)
        assert pk.plan_info(n, h, w)["matrix_path"] == 0
        compare(d, run_gpu(pk, d.x, d.bias, True))
        y = run_gpu(pk, d.x, None, False)
        compare(d, y, bias=None, relu=False)
        assert np.array_equal(run_gpu(pk, d.x, None, False), y)      # a fixed order of additions
    # another shape of the same handle, unplanned
    d2 = _layer(dtype, 1, ci, co, h + 3, w + 1, stride, lib=lib, seed=5)
    d2.w, d2.pid, d2.masks, d2.bias = d.w, d.pid, d.masks, d.bias
    compare(d2, run_gpu(pk, d2.x, d2.bias, True))


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("stride", [1, 2])
def test_any_four_of_nine_taps(dtype, stride):
    """Masks outside the library run with the table of all 126."""
    d = _layer(dtype, 2, 20, 40, 13, 10, stride, seed=7)
    d.masks = ALL_MASKS
    rng = np.random.default_rng(7)
    d.pid = np.where(d.pid < 0, -1, rng.integers(0, 126, d.pid.shape)).astype(np.int16)
    pk = binding.Packed(20, 40, stride, dtype, d.masks, d.w, d.pid)
    pk.plan(2, 13, 10, splits=1)
    compare(d, run_gpu(pk, d.x, d.bias, True))


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("pool", [0, 2])
@pytest.mark.parametrize("ci,co", [(3, 40), (24, 37)])
def test_fused_operators(dtype, pool, ci, co):
    d = _layer(dtype, 2, ci, co, 14, 22, seed=co + pool)
    pk = pack(d)
    pk.plan(2, 14, 22, splits=1, no_small_blocks=True)
    assert pk.plan_info(2, 14, 22)["matrix_path"] == 0
    res = _residual(d, 14, 22, seed=3)
    compare_fused(d, run_fused(pk, d, True, pool, res), True, pool, res)
    if dtype == "i8":
        scale = (wl.uniform01(4, "AUX", 2, co) * 2e-3 + 1e-4).astype(np.float32)
        compare_fused(d, run_fused(pk, d, True, pool, res, scale, 9), True, pool, res, scale, 9)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("warps", [1, 3, 16])
@pytest.mark.parametrize("m,k,co,br,bc", [
    (1, 8, 8, 8, 8),
    (257, 45, 19, 8, 16),         # odd extents: scalar paths
    (300, 200, 264, 16, 64),      # ragged blocks and tiles, several stages
    (1000, 256, 130, 32, 32),
])
def test_block_pruned_product(dtype, warps, m, k, co, br, bc):
    import torch
    d = wl.make_block_gemm(wl.GemmSpec("t", m, k, co, br, bc, 0.5, 0.5, dtype), seed=m + k)
    g = binding.BlockGemm(k, co, br, bc, dtype, d.w, d.row_keep, d.col_keep, warps_per_block=warps)
    assert g.stats()["device_bytes"] == g.stats()["stream_bytes"]        # no weight image beside the stream
    t = torch.float32 if dtype == "f32" else torch.float16
    ref, S = oracle.block_gemm(d.x, d.w, d.row_keep, d.col_keep, br, bc, bias=d.bias, relu=True, with_scale=True)
    for shift in (0, 1):                                 # tensors that start on an element, not on 16 bytes
        x = torch.zeros(m * k + shift, dtype=t, device="cuda")
        x[shift:] = torch.from_numpy(d.x).cuda().reshape(-1)
        buf, y = guarded_output((m, co), t)
        b = torch.from_numpy(d.bias).cuda()
        g.run(x.data_ptr() + shift * x.element_size(), m, b.data_ptr(), True, y.data_ptr())
        g.sync()
        check_guards(buf)
        assert (np.abs(y.cpu().numpy().astype(np.float64) - ref) <= TOL[dtype] * np.maximum(np.abs(ref), 0.01 * S) + 2.0 ** -25).all()
