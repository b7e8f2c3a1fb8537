"""The extension module's calls give what the ctypes path gives, and leave to that path whatever is not an ordinary call."""
import ctypes
import os
import threading

import pytest
import torch

from paper_1908_05858_b200 import binding as B


@pytest.fixture
def native():
    B.lib()
    return B._native


def test_leaves_everything_but_cuda_tensors_alone(native):
    x, a, w = torch.zeros(1, 64, 4, 4), torch.zeros(1, 4, 4, 1, dtype=torch.int64), torch.zeros(8, 3, 3, 1, dtype=torch.int64)
    v = torch.zeros(8)
    assert native.pack(x, 0) is None and native.pack(None, 0) is None and native.pack(x) is None and native.pack(x, 2.0) is None
    assert native.bconv2d(a, 64, w, (1, 1), (1, 1), -1, 1) is None and native.bconv2d() is None
    assert native.bn_sign_pack(a, 64, w, v, v, (1, 1), (1, 1), -1) is None
    assert native.bn_add_sign_pack(a, 64, w, v, v, x, (1, 1), (1, 1), -1, True) is None
    assert native.tc_bconv2d(a, w, 64, 8, 3, 3, (1, 1), (1, 1), -1, 1) is None
    with pytest.raises(B.DabnnError):
        B.pack(x)
    with pytest.raises(TypeError):
        native.bind(1)


def test_the_library_loads_without_the_module(native, monkeypatch, tmp_path):
    """The module is a faster way to make the same calls: missing, or not loadable, it leaves them to ctypes."""
    broken = tmp_path / os.path.basename(B.native_path())
    broken.write_bytes(b"not a shared object")
    for path in (str(tmp_path / ("absent" + broken.name)), str(broken)):
        monkeypatch.setattr(B, "native_path", lambda: path)
        monkeypatch.setattr(B, "_lib", None)
        monkeypatch.setattr(B, "_native", native)
        with pytest.warns(RuntimeWarning, match="ctypes"):
            assert B.lib().dabnn_words_per_pixel(65) == 2
        assert B._native is None
        with pytest.raises(B.DabnnError):
            B.pack(torch.zeros(1, 64, 4, 4))


def test_the_module_of_another_torch_or_interpreter_is_not_taken(native, monkeypatch):
    from paper_1908_05858_b200 import build

    path = B.native_path()
    assert os.path.exists(path) and build.build_native() == path
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    assert not os.path.exists(B.native_path())
    monkeypatch.undo()
    monkeypatch.setattr(B.sysconfig, "get_config_var", lambda name: ".cpython-399.so")
    assert not os.path.exists(B.native_path())


def general(f):
    """f() with an allocator of the caller's own: the ctypes path."""
    prev = B.set_output_allocator(lambda shape, dtype, device: torch.empty(shape, dtype=dtype, device=device))
    try:
        return f()
    finally:
        B.set_output_allocator(prev)


def plain(f):
    prev = B.set_output_allocator(None)
    try:
        return f()
    finally:
        B.set_output_allocator(prev)


def same(f):
    want, got = general(f), plain(f)
    want, got = (t if isinstance(t, tuple) else (t,) for t in (want, got))
    torch.cuda.synchronize()
    for p, q in zip(want, got, strict=True):
        assert (p is None and q is None) or (p.dtype == q.dtype and p.shape == q.shape and p.stride() == q.stride() and torch.equal(p, q))
    return got


@pytest.mark.gpu
@pytest.mark.parametrize("N,C,H,W,O,k,stride", [(1, 64, 14, 14, 64, 3, 1), (3, 100, 9, 7, 70, 3, 2), (2, 512, 5, 6, 33, 1, 1), (40, 128, 14, 14, 128, 3, 1)])
def test_same_as_the_general_path(native, N, C, H, W, O, k, stride):
    g = torch.Generator(device="cuda")
    g.manual_seed(C)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    x, w = rnd(N, C, H, W), plain(lambda: B.pack_weights(rnd(O, C, k, k)))
    geom = ((stride, stride), (k // 2, k // 2), -1)
    a = same(lambda: B.pack(x))[0]
    same(lambda: B.pack(x.permute(0, 2, 3, 1).contiguous(), B.NHWC))
    same(lambda: B.pack(x.permute(0, 2, 3, 1), B.NHWC))               # not contiguous
    same(lambda: B.pack(x[:, :, ::1, : W - 1]))                       # a slice
    same(lambda: B.pack(torch.nn.Parameter(x)))
    assert native.pack(x, 0) is not None and native.pack(x[:, :, :, : W - 1], 0) is None
    scale, shift = rnd(O), rnd(O)
    for pad_value in (-1, 1):
        gm = geom[:2] + (pad_value,)
        for layout in (B.NHWC, B.NCHW):
            out = same(lambda: B.bconv2d(a, C, w, *gm, out_layout=layout))[0]
        same(lambda: B.bconv2d_bn_sign_pack(a, C, w, scale, shift, *gm))
    assert native.bconv2d(a, C, w, *geom, 1) is not None
    same(lambda: B.bconv2d(a, C, w, list(geom[0]), list(geom[1]), -1))  # lists: the general path
    same(lambda: B.bconv2d_bn_sign_pack(a, C, w, torch.stack([scale, shift], 1)[:, 0], shift, *geom))  # a strided vector
    residual = rnd(N, out.shape[2], out.shape[3], O)
    for want_bits in (True, False):
        same(lambda: B.bconv2d_bn_add_sign_pack(a, C, w, scale, shift, residual, *geom, want_bits=want_bits))
    wt = B.TcWeights(w, C)
    same(lambda: B.tc_bconv2d(a, wt, *geom))
    same(lambda: B.tc_bconv2d(a, wt, *geom, out_layout=B.NCHW))
    same(lambda: B.tc_bconv2d_bn_sign_pack(a, wt, scale, shift, *geom))
    same(lambda: B.tc_bconv2d_bn_add_sign_pack(a, wt, scale, shift, residual, *geom))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        same(lambda: B.bconv2d(B.pack(x), C, w, *geom))
    results = [None] * 4
    def work(i):  # noqa: E306
        with torch.cuda.stream(torch.cuda.Stream()):
            results[i] = B.bconv2d(a, C, w, *geom)
            torch.cuda.current_stream().synchronize()
    prev = B.set_output_allocator(None)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in threads], [t.join() for t in threads]
    B.set_output_allocator(prev)
    assert all(torch.equal(r, plain(lambda: B.bconv2d(a, C, w, *geom))) for r in results)


@pytest.mark.gpu
def test_what_was_refused_stays_refused(native):
    x = torch.randn(2, 64, 6, 6, device="cuda")
    a, w = plain(lambda: B.pack(x)), plain(lambda: B.pack_weights(torch.randn(8, 64, 3, 3, device="cuda")))
    v, wt = torch.ones(8, device="cuda"), plain(lambda: B.TcWeights(w, 64))
    calls = [lambda: B.pack(x.double()), lambda: B.pack(x.half()), lambda: B.pack(x[0]), lambda: B.pack(x.cpu()), lambda: B.pack(x[:0]),
             lambda: B.bconv2d(a, 65, w), lambda: B.bconv2d(a, 64, w, (0, 1)), lambda: B.bconv2d(a, 64, w, (1, 1), (0, 0), 0),
             lambda: B.bconv2d(a, 64, w, (1, 1), (2**31 - 1, 2**31 - 1)), lambda: B.tc_bconv2d(a, wt, (1, 1), (2**31 - 1, 2**31 - 1)),
             lambda: B.bconv2d(a, 64, w, (1, 1), (-1, 0)), lambda: B.bconv2d(a.int(), 64, w), lambda: B.bconv2d(a[:, :2, :2].contiguous(), 64, w),
             lambda: B.bconv2d_bn_sign_pack(a, 64, w, v.double(), v), lambda: B.bconv2d_bn_add_sign_pack(a, 64, w, v, v, torch.zeros(2, 4, 4, 7, device="cuda"))]
    for f in calls:
        seen = []
        for path in (general, plain):
            with pytest.raises(Exception) as e:
                path(f)
            seen.append((e.type, str(e.value)))
        assert seen[0] == seen[1]


@pytest.mark.gpu
def test_a_launch_that_failed_is_reported_and_not_made_again(native):
    """The library reads and clears the runtime's last error, so a second call after a failed one could succeed in silence.  With
    entries that only return a status: a failed launch raises, refused arguments go to the general path."""
    x, res, v = torch.randn(2, 64, 6, 6, device="cuda"), torch.randn(2, 6, 6, 8, device="cuda"), torch.ones(8, device="cuda")
    a, w = plain(lambda: B.pack(x)), plain(lambda: B.pack_weights(torch.randn(8, 64, 3, 3, device="cuda")))
    wt, geom = B.TcWeights(w, 64), ((1, 1), (1, 1), -1)
    calls = [lambda: B.pack(x), lambda: B.bconv2d(a, 64, w, *geom), lambda: B.bconv2d_bn_sign_pack(a, 64, w, v, v, *geom),
             lambda: B.bconv2d_bn_add_sign_pack(a, 64, w, v, v, res, *geom), lambda: B.tc_bconv2d(a, wt, *geom),
             lambda: B.tc_bconv2d_bn_sign_pack(a, wt, v, v, *geom), lambda: B.tc_bconv2d_bn_add_sign_pack(a, wt, v, v, res, *geom)]
    want = [general(f) for f in calls]
    made, status = [], [0]
    fake = ctypes.CFUNCTYPE(ctypes.c_int)(lambda: made.append(1) or status[0])
    try:
        native.bind(*[ctypes.cast(fake, ctypes.c_void_p).value] * len(B._NATIVE_ENTRIES), B._check)
        for f, y in zip(calls, want, strict=True):
            for status[0] in (6, 7):  # DABNN_ERR_CUDA, DABNN_ERR_TIMEOUT
                made.clear()
                with pytest.raises(B.DabnnError, match="dabnn status %d" % status[0]):
                    plain(f)
                assert len(made) == 1
            status[0] = 2  # DABNN_ERR_SHAPE
            got = plain(f)
            assert all(torch.equal(p, q) for p, q in zip(*(t if isinstance(t, tuple) else (t,) for t in (got, y)), strict=True))
    finally:
        native.bind(*[ctypes.cast(getattr(B.lib(), name), ctypes.c_void_p).value for name in B._NATIVE_ENTRIES], B._check)
    assert torch.equal(plain(calls[0]), want[0])
