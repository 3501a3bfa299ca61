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


def test_refusals():
    X, R, Ri, Wq, Ws = _layer(4, 256, 64, 1)
    with pytest.raises(ValueError, match="R_inter"):
        torq.torq_rotated_linear(X, R.float(), Ri, Wq, Ws)
    with pytest.raises(ValueError, match="X"):
        torq.torq_rotated_linear(X.t(), R, Ri, Wq, Ws)
    with pytest.raises(ValueError, match="Wq"):
        torq.torq_rotated_linear(X, R, Ri, Wq.cpu(), Ws)
    with pytest.raises(torq.TorqError):                            # from the library: the workspace is too small
        torq.torq_rotated_linear(X, R, Ri, Wq, Ws, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
