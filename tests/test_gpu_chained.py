"""The calls of the C ABI start while the kernel before them drains, and some kernels let their successor in before their own stores.
Every call here reads what such a kernel has just written, in buffers that each step writes again with other values: a read that
does not wait finds the values of the step before."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_1908_05858_b200 import binding

    binding.lib()
    return binding


def stream():
    return torch.cuda.current_stream().cuda_stream


# The convolutions are small enough for the integer pipes, one CTA per SM at most: they let the next kernel in ahead of their stores.
# Between them the cases take every pack kernel, from fp32 and from int32.
CASES = [
    # N, C, H, W, O, k, stride
    (1, 64, 14, 14, 64, 3, 1),   # NCHW in 16-byte pieces, NHWC of whole words
    (1, 64, 7, 7, 64, 3, 1),     # NCHW, 49 pixels: a word's channels as one run
    (1, 100, 9, 7, 70, 3, 2),    # NHWC with a channel tail, stride 2
    (1, 65, 7, 5, 70, 3, 1),     # NCHW pixel by pixel: 65 x 35 values are no multiple of 4
    (2, 33, 6, 6, 20, 1, 1),     # NHWC, short rows: a thread per word
    (1, 512, 4, 4, 448, 3, 2),   # words of a pixel split among CTAs
]


@pytest.mark.parametrize("N,C,H,W,O,k,stride", CASES)
def test_a_chain_of_calls_gives_what_they_give_one_by_one(B, N, C, H, W, O, k, stride):
    L, pad = B.lib(), k // 2
    OH, OW, words, owords, STEPS = B.out_dim(H, k, stride, pad), B.out_dim(W, k, stride, pad), (C + 63) // 64, (O + 63) // 64, 5
    g = torch.Generator(device="cuda")
    g.manual_seed(C)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    xs, ws, bns = [rnd(N, C, H, W) for _ in range(STEPS)], [rnd(O, C, k, k) for _ in range(STEPS)], [rnd(O).abs() + 0.5 for _ in range(STEPS)]
    w2, v2 = B.pack_weights(rnd(24, O, 1, 1)), rnd(24)
    new = lambda dtype, *s: torch.zeros(s, dtype=dtype, device="cuda")  # noqa: E731
    i64, i32, f32 = torch.int64, torch.int32, torch.float32
    x, w, wt = new(f32, N, C, H, W), new(i64, O, k, k, words), B.TcWeights(B.pack_weights(ws[0]), C)
    scale, shift, res, res2 = new(f32, O), new(f32, O), rnd(N, OH, OW, O), rnd(N, OH, OW, 24)
    packed = lambda c=O: new(i64, N, OH, OW, (c + 63) // 64)  # noqa: E731
    out = {"a": new(i64, N, H, W, words), "sums": new(i32, N, OH, OW, O), "sums_nchw": new(i32, N, O, OH, OW), "tc_sums": new(i32, N, OH, OW, O),
           "y": new(f32, N, OH, OW, O), "y2": new(f32, N, OH, OW, 24), "tc_y": new(f32, N, OH, OW, O)}
    out.update({name: packed() for name in ("of_sums", "of_nchw", "y_bits", "of_y", "of_y_nchw", "signs", "tc_signs", "tc_y_bits")})
    out.update(y2_bits=packed(24), of_y_c2=new(i64, N, (O + 127) // 128, OH, OW, 2), from_c2=new(i32, N, OH, OW, 24))
    seen = [{name: torch.zeros_like(t) for name, t in out.items()} for _ in range(STEPS)]
    p = lambda name: out[name].data_ptr()  # noqa: E731
    shape, cv = B.Shape(N, C, H, W), B._conv(k, k, (stride, stride), (pad, pad), -1)
    shape2, cv2 = B.Shape(N, O, OH, OW), B._conv(1, 1, (1, 1), (0, 0), -1)
    nhwc, nchw, geom = B.NHWC, B.NCHW, ((stride, stride), (pad, pad), -1)

    def run(sync):
        def call(status, *_):
            assert status in (0, None)
            if sync:
                torch.cuda.synchronize()

        for i in range(STEPS):
            x.copy_(xs[i])
            call(L.dabnn_pack_weights(ws[i].data_ptr(), O, C, k, k, w.data_ptr(), stream()))
            call(None, B.pack(x, out=out["a"]))
            call(None, B.bconv2d(out["a"], C, w, *geom, out=out["sums"]))
            call(None, B.pack_i32(out["sums"], nhwc, out=out["of_sums"]))
            call(None, B.bconv2d(out["a"], C, w, *geom, nchw, out=out["sums_nchw"]))
            call(None, B.pack_i32(out["sums_nchw"], out=out["of_nchw"]))
            call(L.dabnn_bn_fold(*[bns[(i + q) % STEPS].data_ptr() for q in (0, 1, 2, 3)], 1e-5, O, scale.data_ptr(), shift.data_ptr(), stream()))
            call(L.dabnn_bconv2d_bn_add_sign_pack(p("a"), shape, w.data_ptr(), O, cv, scale.data_ptr(), shift.data_ptr(), res.data_ptr(),
                                                  p("y"), p("y_bits"), stream()))
            call(None, B.pack(out["y"], nhwc, out=out["of_y"]))
            call(None, B.bconv2d_bn_sign_pack(out["a"], C, w, scale, shift, *geom, out=out["signs"]))
            # (the packed signs of the call before as activations, residual form)
            call(L.dabnn_bconv2d_bn_add_sign_pack(p("signs"), shape2, w2.data_ptr(), 24, cv2, v2.data_ptr(), v2.data_ptr(), res2.data_ptr(),
                                                  p("y2"), p("y2_bits"), stream()))
            call(L.dabnn_tc_prepare_weights(w.data_ptr(), O, C, k, k, wt.buf.data_ptr(), stream()))
            call(None, B.tc_bconv2d(out["a"], wt, *geom, out=out["tc_sums"]))
            call(None, B.tc_bconv2d_bn_sign_pack(out["a"], wt, scale, shift, *geom, out=out["tc_signs"]))
            call(L.dabnn_bconv2d_bn_add_sign_pack(p("a"), shape, w.data_ptr(), O, cv, scale.data_ptr(), shift.data_ptr(), out["y"].data_ptr(),
                                                  p("y"), p("y_bits"), stream()))  # (in place, on what the pack above has read)
            call(None, B.pack(out["y"].view(N, O, OH, OW), out=out["of_y_nchw"]))  # (the same values taken as NCHW)
            call(L.dabnn_tc_bconv2d_bn_add_sign_pack(p("a"), shape, wt.buf.data_ptr(), O, cv, scale.data_ptr(), shift.data_ptr(), p("y"),
                                                     p("tc_y"), p("tc_y_bits"), stream()))
            call(None, B.pack_as(out["y"], B.PACKED_NC1HWC2, nhwc, out=out["of_y_c2"]))
            call(None, B.bconv2d_from(out["of_y_c2"], B.PACKED_NC1HWC2, O, w2, out=out["from_c2"]))
            for name, t in out.items():
                seen[i][name].copy_(t)

    def collect():
        torch.cuda.synchronize()
        got = [{name: t.clone() for name, t in step.items()} for step in seen]
        for step in seen:
            for t in step.values():
                t.zero_()
        return got

    def same(got, want):
        for i, (q, r) in enumerate(zip(got, want, strict=True)):
            for name in out:
                assert torch.equal(q[name], r[name]), (i, name)

    run(True)
    want = collect()
    assert all(torch.equal(s["tc_sums"], s["sums"]) and torch.equal(s["tc_signs"], s["signs"]) and torch.equal(s["of_nchw"], s["of_sums"]) for s in want)
    assert all(not torch.equal(want[i]["sums"], want[i - 1]["sums"]) for i in range(STEPS))
    for _ in range(4):
        run(False)
        same(collect(), want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(False)
    for _ in range(3):
        graph.replay()
        same(collect(), want)
    del graph
    assert B.last_device_flag() == 0


@pytest.mark.parametrize("captured", [False, True])
def test_a_call_behind_a_join_waits_for_both_streams(B, captured):
    """A pack whose input another stream's convolution writes, with a convolution of its own stream just before it."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    N, C, HW, O, STEPS = 1, 64, 14, 64, 6
    a, w = [B.pack(rnd(N, C, HW, HW)) for _ in range(STEPS)], [B.pack_weights(rnd(O, C, 3, 3)) for _ in range(STEPS)]
    here, there = (torch.zeros((N, HW, HW, O), dtype=torch.int32, device="cuda") for _ in range(2))
    bits = [torch.zeros((N, HW, HW, 1), dtype=torch.int64, device="cuda") for _ in range(2 * STEPS)]
    side = torch.cuda.Stream()

    def run(sync):
        main = torch.cuda.current_stream()
        for i in range(STEPS):
            side.wait_stream(main)
            with torch.cuda.stream(side):
                B.bconv2d(a[i], C, w[i], (1, 1), (1, 1), -1, out=there)
            B.bconv2d(a[i], C, w[(i + 1) % STEPS], (1, 1), (1, 1), -1, out=here)
            main.wait_stream(side)
            if sync:
                torch.cuda.synchronize()
            B.pack_i32(there, B.NHWC, out=bits[2 * i])
            B.pack_i32(here, B.NHWC, out=bits[2 * i + 1])
            if sync:
                torch.cuda.synchronize()

    run(True)
    want = [t.clone() for t in bits]
    graph = None
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(False)
    for _ in range(5):
        for t in bits:
            t.zero_()
        graph.replay() if captured else run(False)
        torch.cuda.synchronize()
        assert all(torch.equal(p, q) for p, q in zip(bits, want, strict=True))
    assert not torch.equal(want[0], want[2])
