"""The native marshalling of the layer calls: the same results as the two kernels called one by one, on the current
stream, on a given stream and from two threads at once; operands that it does not take are refused by name as before."""
import threading

import pytest
import torch

from paper_2605_19561_b200 import torq

pytestmark = pytest.mark.gpu


def _layer(M, d, N, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = (torch.randn(M, d, device="cuda", generator=g) * 2).bfloat16()
    R = (torch.randn(d, d, device="cuda", generator=g) / d ** 0.5).bfloat16()
    Ri = (torch.randn(d // 32, 32, 32, device="cuda", generator=g) / 32 ** 0.5).bfloat16()
    Wq = torch.randint(0, 256, (N, d // 2), dtype=torch.uint8, device="cuda", generator=g)
    Ws = torch.randint(120, 132, (torq.torq_scales_bytes(N, d),), dtype=torch.uint8, device="cuda", generator=g)
    return X, R, Ri, Wq, Ws


def test_streams_and_threads():
    ops = [_layer(40, 512, 264, s) for s in range(2)]
    ref = []
    for X, R, Ri, Wq, Ws in ops:
        c, s = torq.torq_rotate_quantize(X, R, Ri)
        ref.append(torq.torq_mxfp4_gemm(c, s, Wq, Ws))
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    got = torq.torq_rotated_linear(*ops[0], stream=st)             # a given stream
    with torch.cuda.stream(st):
        got2 = torq.torq_rotated_linear(*ops[1])                   # the current stream
    st.synchronize()
    assert torch.equal(got, ref[0]) and torch.equal(got2, ref[1])
    out = [None, None]

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(50):
                out[i] = torq.torq_rotated_linear(*ops[i])
            torch.cuda.current_stream().synchronize()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
    assert torq.torq_last_device_error() == 0


def test_refusals(binding):
    X, R, Ri, Wq, Ws = _layer(4, 256, 64, 1)
    with pytest.raises(ValueError, match="R_inter"):
        torq.torq_rotated_linear(X, R.float(), Ri, Wq, Ws)
    with pytest.raises(ValueError, match="X"):
        torq.torq_rotated_linear(X.t(), R, Ri, Wq, Ws)
    with pytest.raises(ValueError, match="Wq"):
        torq.torq_rotated_linear(X, R, Ri, Wq.cpu(), Ws)
    with pytest.raises(torq.TorqError):                            # from the library: the workspace is too small
        torq.torq_rotated_linear(X, R, Ri, Wq, Ws, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))


@pytest.fixture(params=["native", "ctypes"])
def binding(request, monkeypatch):
    """Both ways a layer call can take: the native binding, and ctypes where that is missing."""
    if request.param == "ctypes":
        monkeypatch.setattr(torq, "_layer", torq._layer_ctypes)
    else:
        monkeypatch.setattr(torq, "_layer", torq._layer_native())
        assert torq._layer is not None


def _layer_calls():
    """Every whole-layer entry point as f(X, Y=..., workspace=...), with the operands it takes."""
    X, R, Ri, Wq, Ws = _layer(4, 256, 64, 1)
    Rb, Rs = R[:8, :8].contiguous(), Ri[0].contiguous()
    Ws16 = torch.full((torq.torq_nvfp4_scales_bytes(64, 256),), 0x38, dtype=torch.uint8, device="cuda")
    W8 = torch.zeros(64, 256, dtype=torch.uint8, device="cuda")
    return X, {
        "mxfp4": lambda **k: torq.torq_rotated_linear(X, R, Ri, Wq, Ws, **k),
        "structured": lambda **k: torq.torq_rotated_linear_structured(X, Rb, Rs, Wq, Ws, **k),
        "nvfp4": lambda **k: torq.torq_rotated_linear_nvfp4(X, R, Ri, 0.01, Wq, Ws16, 0.01, **k),
        "mxint4": lambda **k: torq.torq_rotated_linear_mxint4(X, R, Ri, W8, Ws, **k),
    }


@pytest.mark.parametrize("kind", ["mxfp4", "structured", "nvfp4", "mxint4"])
def test_results_and_scratch_that_are_refused(binding, kind):
    """A result that could not hold what the kernels write, or scratch that they could not use: ValueError, nothing launched,
    nothing written."""
    X, calls = _layer_calls()
    call = calls[kind]
    torch.cuda.synchronize()
    before = torq.torq_launch_count()
    wide = torch.full((4, 80), 7.0, dtype=torch.bfloat16, device="cuda")
    half = torch.full((4, 64), 7.0, dtype=torch.float16, device="cuda")
    small = torch.full((3, 64), 7.0, dtype=torch.bfloat16, device="cuda")
    for Y in (wide[:, :64], half, small, torch.empty(4, 64, dtype=torch.bfloat16), torch.empty(4, 64, dtype=torch.int16, device="cuda")):
        with pytest.raises(ValueError, match="Y"):
            call(Y=Y)
    size = 1 << 20
    for ws in (torch.empty(size, dtype=torch.uint8), torch.empty(2 * size, dtype=torch.uint8, device="cuda")[::2]):
        with pytest.raises(ValueError, match="workspace"):
            call(workspace=ws)
    with pytest.raises(ValueError):
        call(out_dtype=torch.float16)
    torch.cuda.synchronize()
    assert torq.torq_launch_count() == before
    assert bool((wide == 7).all()) and bool((half == 7).all()) and bool((small == 7).all())


@pytest.mark.parametrize("kind", ["mxfp4", "structured", "nvfp4", "mxint4"])
def test_results_and_scratch_that_are_taken(binding, kind):
    """As before: a larger or differently shaped contiguous result, scratch of any type (one byte counted per element)."""
    X, calls = _layer_calls()
    call = calls[kind]
    ref = call()
    big = torch.full((6, 64), 7.0, dtype=torch.bfloat16, device="cuda")
    call(Y=big)
    flat = call(Y=torch.empty(4 * 64, dtype=torch.bfloat16, device="cuda"), workspace=torch.empty(1 << 20, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    assert torch.equal(big[:4], ref) and bool((big[4:] == 7).all()) and torch.equal(flat.view(4, 64), ref)


def test_the_separate_gemms_refuse_the_same_results():
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randint(0, 256, (4, 128), dtype=torch.uint8, device="cuda", generator=g)
    W = torch.randint(0, 256, (64, 128), dtype=torch.uint8, device="cuda", generator=g)
    s = torch.full((torq.torq_nvfp4_scales_bytes(64, 256),), 0x38, dtype=torch.uint8, device="cuda")
    before = torq.torq_launch_count()
    for Y in (torch.empty(4, 64, dtype=torch.float16, device="cuda"), torch.empty(3, 64, dtype=torch.bfloat16, device="cuda")):
        for f in (lambda: torq.torq_mxfp4_gemm(A, s, W, s, Y=Y), lambda: torq.torq_nvfp4_gemm(A, s, 1.0, W, s, 1.0, Y=Y),
                  lambda: torq.torq_mxint4_gemm(A, s, W, s, Y=Y)):
            with pytest.raises(ValueError, match="Y"):
                f()
    assert torq.torq_launch_count() == before
