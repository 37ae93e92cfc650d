"""What the host code does when a CUDA call fails, and what a handle holds: the library's own objects
linked with a stand-in for the CUDA runtime (fake_cuda.cpp), run in a process of its own."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2206_10620_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    build.build()
    objs = [os.path.join(build._OBJ_DIR, os.path.splitext(s)[0] + ".o") for s in build._SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libpatconv_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           os.path.join(HERE, "fake_cuda.cpp")] + objs + ["-o", out])
    return out


PRELUDE = """
import ctypes, os
import numpy as np
from paper_2206_10620_b200 import binding, workloads as wl
fake = ctypes.CDLL(os.environ["XGEN_PATCONV_LIB"])
fake.fake_live_bytes.restype = fake.fake_launch.restype = ctypes.c_longlong
binding.lib()

def conv(dtype, ci, co, stride=1, prune=0.5, device=0):
    d = wl.make_layer(wl.LayerSpec("t", 1, ci, co, 4, 4, stride, dtype, prune, 12, "he", "u01", 0.05, True, 0), seed=1)
    return binding.Packed(ci, co, stride, dtype, d.masks, d.w, d.pid, device=device)

def gemm(dtype, k, co, **kw):
    d = wl.make_block_gemm(wl.GemmSpec("t", 4, k, co, 16, 16, 0.5, 0.5, dtype), seed=1)
    return binding.BlockGemm(k, co, 16, 16, dtype, d.w, d.row_keep, d.col_keep, **kw)

def status(call, *a, **kw):
    try:
        call(*a, **kw)
    except binding.PatconvError as e:
        return e.status
    return 0

X, Y, B = 1 << 40, 2 << 40, 3 << 40          # addresses of tensors that nothing reads
"""


def _run(fake_lib, code):
    env = dict(os.environ, XGEN_PATCONV_LIB=fake_lib, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code)], env=env, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("dtype,ci", [("f16", 64), ("i8", 128)])
def test_a_tensor_map_that_cannot_be_made_is_an_error(fake_lib, dtype, ci):
    """A plan for copied rows holds no table for gathered ones, so the launch must not fall back to them."""
    _run(fake_lib, """
        pk = conv(%r, %d, 64)
        run = lambda: status(pk.run, X, 2, 20, 20, B, True, Y)
        assert run() == 0 and fake.fake_launches() > 0
        n = fake.fake_launches()
        fake.fake_fail_encode(1)             # (the plan, with the map of the weights, is kept: this is x's)
        assert run() == 6 and fake.fake_launches() == n
        assert run() == 0 and fake.fake_launches() == n + 1
    """ % (dtype, ci))


def test_an_upload_that_fails_half_way_leaves_nothing(fake_lib):
    """The block-pruned product's command stream, uploaded by the first run that needs it: a run after a
    failed one uploads again."""
    _run(fake_lib, """
        g = gemm("f32", 64, 48)
        run = lambda: status(g.run, X, 32, B, True, Y)
        held, n = fake.fake_live_bytes(), fake.fake_launches()
        for nth in (1, 2):
            fake.fake_fail_encode(1)         # the matrix path cannot run, so the stream is asked for
            fake.fake_fail_alloc(nth)
            assert run() == 5 and fake.fake_launches() == n and fake.fake_live_bytes() == held
        fake.fake_fail_encode(1)
        assert run() == 0 and fake.fake_launches() == n + 1 and fake.fake_live_bytes() > held
    """)


def test_a_handle_holds_its_weight_image_and_no_more(fake_lib):
    """The scratch of the upload is shared, 1 MB while there is any handle; a failed upload leaves nothing."""
    _run(fake_lib, """
        assert fake.fake_live_bytes() == 0
        for nth in (1, 2, 3):
            fake.fake_fail_alloc(nth)
            assert status(conv, "f32", 16, 32) == 5 and fake.fake_live_bytes() == 0
        first = gemm("f16", 32, 32)
        assert fake.fake_live_bytes() <= (1 << 20) + 2 * 32 * 32 + 64
        round16 = lambda n: -(-n // 16) * 16
        for dtype, ci, co in (("f32", 16, 32), ("f32", 300, 260), ("f16", 300, 260), ("i8", 300, 260)):
            per, parts = {"f32": (8, 3), "f16": (8, 1), "i8": (16, 1)}[dtype]
            image = -(-ci // (2 * per)) * 2 * 9 * parts * round16(co) * 16
            held = fake.fake_live_bytes()
            pk = conv(dtype, ci, co)
            assert image < fake.fake_live_bytes() - held <= image + 64, (dtype, fake.fake_live_bytes() - held - image)
            pk.close()
            assert fake.fake_live_bytes() == held
        for dtype, k, co in (("f32", 700, 500), ("f16", 33, 31)):
            image = -(-k // 16) * 2 * {"f32": 3, "f16": 1}[dtype] * round16(co) * 16
            held = fake.fake_live_bytes()
            g = gemm(dtype, k, co)
            assert image < fake.fake_live_bytes() - held <= image + 64
            g.close()
            fake.fake_fail_alloc(1)
            assert status(gemm, dtype, k, co) == 5 and fake.fake_live_bytes() == held
        first.close()
        assert fake.fake_live_bytes() == 0
    """)


def test_queries_tell_of_what_runs_and_what_is_held(fake_lib):
    """xgen_patconv_plan_info's matrix_* fields are the launch of a run, device_bytes is what was allocated."""
    _run(fake_lib, """
        keep = gemm("f16", 32, 32)                # (the shared scratch is there)
        for dtype in ("f32", "f16", "i8"):
            for n, ci, co, h, w in ((1, 16, 32, 8, 8), (40, 64, 64, 40, 40), (32, 256, 256, 28, 28), (1, 512, 96, 14, 14), (3, 67, 93, 45, 77)):
                held = fake.fake_live_bytes()
                pk = conv(dtype, ci, co)
                pk.plan(n, h, w)
                info, st = pk.plan_info(n, h, w), pk.stats()
                assert info["matrix_path"] == 1 and st["image_bytes"] > 0
                assert st["device_bytes"] == fake.fake_live_bytes() - held
                pk.run(X, n, h, w, B, True, Y)
                got = [info["matrix_" + k] for k in ("blocks", "threads", "shared_bytes", "cluster")]
                assert got == [fake.fake_launch(i) for i in range(4)], (got, dtype, n, ci, co, h, w)
                pk.plan(n, h, w, splits=2)
                info = pk.plan_info(n, h, w)
                pk.run(X, n, h, w, B, True, Y)
                assert info["matrix_path"] == 0 == info["matrix_blocks"]
                assert [info["blocks"], info["threads_per_block"], info["shared_bytes"]] == [fake.fake_launch(i) for i in range(3)]
                assert pk.stats()["device_bytes"] == fake.fake_live_bytes() - held
                pk.close()
        pk = conv("f32", 16, 32, device=-1)
        assert pk.stats()["device_bytes"] == 0 and pk.plan_info(1, 8, 8)["matrix_path"] == 0
        for kw in ({}, {"warps_per_block": 4}):
            held = fake.fake_live_bytes()
            g = gemm("f16", 200, 70, **kw)
            assert g.stats()["device_bytes"] == fake.fake_live_bytes() - held
            g.close()
    """)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i8"])
@pytest.mark.parametrize("stride", [1, 2])
def test_every_layer_of_the_matrix_path_has_a_plan(fake_lib, dtype, stride):
    """No shape falls back to the command stream: whatever its rows, tiles, batch and fused operators are, a run launches the
    matrix kernel and allocates nothing."""
    _run(fake_lib, """
        dtype, stride = %r, %d
        threads = {"f32": 16, "f16": 24, "i8": 24}[dtype] * 32
        for ci in (8, 17, 33, 67, 128, 131, 503):
            for co in (16, 37, 93, 256, 400):
                pk = conv(dtype, ci, co, stride)
                for n, h, w in ((1, 1, 1), (1, 14, 14), (1, 57, 57), (4, 224, 224), (32, 56, 56), (8, 112, 112), (64, 28, 28), (200, 7, 7), (2, 200, 111), (3, 5, 700)):
                    if n * h * w * max(ci, co) >= 2 ** 31:
                        continue
                    held, launches = fake.fake_live_bytes(), fake.fake_launches()
                    ho, wo = pk.out_shape(h, w)
                    pool = 2 if ho %% 2 == 0 and wo %% 2 == 0 else 0
                    assert pk.plan_info(n, h, w)["matrix_path"] == 1, (ci, co, n, h, w)
                    calls = [lambda: pk.run(X, n, h, w, B, True, Y), lambda: pk.run_fused(X, n, h, w, B, Y, residual_ptr=3 << 41),
                             lambda: pk.run_fused(X, n, h, w, B, Y, pool=pool, residual_ptr=3 << 41)]
                    if dtype == "i8":
                        calls.append(lambda: pk.run_fused(X, n, h, w, B, Y, residual_ptr=3 << 41, requant_scale_ptr=B))
                    for call in calls:
                        call()
                        assert fake.fake_launch(1) == threads, (ci, co, n, h, w)
                    assert fake.fake_live_bytes() == held and fake.fake_launches() == launches + len(calls)
                pk.close()
    """ % (dtype, stride))


def test_the_stream_of_a_layer_without_a_plan_is_uploaded_where_it_may_be(fake_lib):
    """The command stream that a run falls back to goes to the handle's device, whichever is current, and never
    from inside a capture or a call that promises not to allocate."""
    _run(fake_lib, """
        for pk, run in ((conv("f16", 33, 48, 2, device=1), lambda p: status(p.run, X, 2, 20, 20, B, True, Y)),
                        (gemm("f32", 64, 48, device=1), lambda p: status(p.run, X, 32, B, True, Y))):
            held, n = fake.fake_live_bytes(), fake.fake_launches()
            fake.fake_capture(1)
            fake.fake_fail_encode(1)             # the matrix path has no plan
            assert run(pk) == 4 and fake.fake_launches() == n and fake.fake_live_bytes() == held
            fake.fake_capture(0)
            if hasattr(pk, "run_static_scratch"):
                fake.fake_fail_encode(1)
                assert status(pk.run_static_scratch, X, 2, 20, 20, B, True, Y, 1) == 4
                assert fake.fake_launches() == n and fake.fake_live_bytes() == held
            fake.fake_fail_encode(1)
            assert fake.fake_device() == 0 and run(pk) == 0 and fake.fake_device() == 0
            assert fake.fake_alloc_device() == 1 and fake.fake_launches() == n + 1 and fake.fake_live_bytes() > held
            pk.close()
    """)


def test_a_plan_uploads_the_stream_where_there_are_no_tensor_maps(fake_lib):
    _run(fake_lib, """
        fake.fake_no_encode(1)
        pk = conv("f16", 64, 48, device=1)
        pk.plan(2, 20, 20)
        assert fake.fake_alloc_device() == 1
        held, n = fake.fake_live_bytes(), fake.fake_launches()
        fake.fake_capture(1)
        assert status(pk.run, X, 2, 20, 20, B, True, Y) == 0
        assert status(pk.run_static_scratch, X, 2, 20, 20, B, True, Y, 1) == 0
        assert fake.fake_launches() == n + 2 and fake.fake_live_bytes() == held
    """)


def test_layers_of_a_few_channels_take_the_faster_kernel(fake_lib):
    """Large images of which little is left, and filters that do not fill the dense kernel's warps: the command stream; small
    images, stride 2 and whole layers: the dense kernel, and always where nothing may be allocated."""
    _run(fake_lib, """
        for dtype, ci, co, n, hw, prune, stride, stream in (
                ("f32", 4, 48, 9, 224, 0.0, 1, True), ("f32", 4, 96, 9, 224, 0.0, 1, True), ("f32", 4, 80, 1, 224, 0.9, 1, True),
                ("f32", 4, 64, 9, 224, 0.9, 1, True), ("f16", 7, 80, 1, 224, 0.9, 1, True), ("i8", 7, 48, 9, 224, 0.9, 1, True),
                ("f32", 3, 64, 1, 224, 0.0, 1, False), ("f32", 3, 64, 9, 224, 0.0, 1, False), ("f16", 3, 32, 9, 224, 0.0, 1, False),
                ("f32", 4, 48, 1, 60, 0.9, 1, False), ("i8", 3, 64, 4, 224, 0.5, 1, False), ("f16", 7, 80, 4, 224, 0.9, 2, False)):
            pk = conv(dtype, ci, co, stride, prune)
            n0 = fake.fake_launches()
            for _ in range(2):                       # weighed, and from the cache
                assert pk.plan_info(n, hw, hw)["few_channel_path"] == int(not stream)
                pk.run(X, n, hw, hw, B, True, Y)
                assert (fake.fake_launch(1) != 128) == stream, (dtype, ci, co, n, hw, prune, stride)
            pk.run_static_scratch(X, n, hw, hw, B, True, Y, 1)
            assert fake.fake_launch(1) == 128 and fake.fake_launches() == n0 + 3
            pk.plan(n, hw, hw, splits=1)             # the caller asks for the stream
            pk.run(X, n, hw, hw, B, True, Y)
            assert fake.fake_launch(1) != 128 and pk.plan_info(n, hw, hw)["few_channel_path"] == 0
            pk.close()
        for handle in (conv("f32", 16, 32), conv("f32", 3, 32, device=-1)):
            assert handle.plan_info(1, 224, 224)["few_channel_path"] == 0
    """)
