"""The give-up path of the bounded device waits, run once on purpose.  Every wait inside the
tensor-core kernels is bounded: when it runs out it latches TORQ_ERR_TIMEOUT with the id of the wait
site, raises the CTA's abort flag, the other roles leave their loops, the kernel drains and returns.
A healthy run never gets there, so torq_selftest_wait_timeout makes a wait run out harmlessly (a
barrier nothing arrives on, a limit of a millisecond): nothing faults, traps or hangs."""
import ctypes

import pytest
import torch

from helpers import captured_launches
from paper_2605_19561_b200 import torq

pytestmark = pytest.mark.gpu

TORQ_ERR_TIMEOUT, SITE_SELFTEST = 6, 7


def test_a_wait_that_runs_out_latches_the_error_word_and_the_library_stays_usable():
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0
    res = torq.torq_selftest_wait_timeout(1_000_000)            # 1 ms
    torch.cuda.synchronize()
    gave_up, left_by_flag, waited_ns = (int(v) for v in res.cpu())
    assert gave_up == 1 and left_by_flag == 1
    assert 500_000 <= waited_ns <= 500_000_000                    # about the limit, far below the 2 s of its own
    err = torq.torq_last_device_error()
    assert err & 0xFF == TORQ_ERR_TIMEOUT and (err >> 8) & 0xFF == SITE_SELFTEST
    assert torq.torq_last_device_error() == 0                     # reading clears it
    # the next ordinary call runs and reports nothing
    z = torch.randn((64, 256), device="cuda")
    codes, scales = torq.torq_quantize_mxfp4(z)
    X = torch.randn((256, 256), device="cuda").to(torch.bfloat16)
    R = torch.eye(256, device="cuda").to(torch.bfloat16)
    c2, s2 = torq.torq_rotate_quantize(X, R, None)
    c3, s3 = torq.torq_rotate_quantize(X, None, None)
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0
    assert torch.equal(c2, c3) and torch.equal(s2, s3)            # identity rotation = quantize-only


def test_argument_errors_launch_nothing():
    before = torq.torq_launch_count()
    L = torq.lib()
    out = torch.zeros(4, dtype=torch.int64, device="cuda")
    import ctypes
    assert L.torq_selftest_wait_timeout(10, ctypes.c_void_p(out.data_ptr()), None) == 2
    assert L.torq_selftest_wait_timeout(1_000_000, None, None) == 1
    assert torq.torq_launch_count() == before


SLOW_KERNEL = rb"""
extern "C" __global__ void slow(unsigned long long ns) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  unsigned long long start, now;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(start));
  for (int i = 0; i < 60000; ++i) {
    __nanosleep(100000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (now - start >= ns) break;
  }
}
"""


def _slow_kernel():
    """launch(ns): one thread on the current stream that lets the next kernel start at once and then sleeps for `ns`."""
    from cuda.bindings import driver as cu, nvrtc

    def ok(res):
        assert int(res[0]) == 0, res[0]
        return res[1] if len(res) == 2 else res[1:]

    prog = ok(nvrtc.nvrtcCreateProgram(SLOW_KERNEL, b"slow.cu", 0, [], []))
    ok(nvrtc.nvrtcCompileProgram(prog, 1, [b"--gpu-architecture=sm_100a"]))
    image = b" " * ok(nvrtc.nvrtcGetCUBINSize(prog))
    ok(nvrtc.nvrtcGetCUBIN(prog, image))
    torch.cuda.synchronize()
    fn = ok(cu.cuModuleGetFunction(ok(cu.cuModuleLoadData(image)), b"slow"))
    return lambda ns: ok(cu.cuLaunchKernel(fn, 1, 1, 1, 1, 1, 1, 0, torch.cuda.current_stream().cuda_stream,
                                           ((ns,), (ctypes.c_uint64,)), 0))


def test_a_slow_kernel_before_is_not_counted_on_the_waits():
    """A kernel that lets its dependents start and then runs longer than the limit of a wait: the call behind it gives the same
    result as by itself and reports nothing.  Pair and one-wave kernels, which start their weights' loads before it has completed."""
    slow = _slow_kernel()
    g = torch.Generator(device="cuda").manual_seed(2)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    for kernel, M, d, N in (("rotate_quantize_pair", 2048, 4096, 0), ("rotate_quantize_wide", 300, 1024, 0),
                            ("mxfp4_gemm_pair", 2048, 4096, 6144), ("mxfp4_gemm_wide", 200, 4096, 6144)):
        if N == 0:
            X, R, out = rnd(M, d), rnd(d, d), [torch.empty(M, d // 2, dtype=torch.uint8, device="cuda"),
                                               torch.empty(torq.torq_scales_bytes(M, d), dtype=torch.uint8, device="cuda")]
            call = lambda: torq.torq_rotate_quantize(X, R, None, out_codes=out[0], out_scales=out[1])
        else:
            A, W = (torch.randint(0, 256, (r, d // 2), generator=g, device="cuda", dtype=torch.uint8) for r in (M, N))
            As, Ws = (torch.full((torq.torq_scales_bytes(r, d),), 127, dtype=torch.uint8, device="cuda") for r in (M, N))
            out = [torch.empty(M, N, dtype=torch.float32, device="cuda")]
            call = lambda: torq.torq_mxfp4_gemm(A, As, W, Ws, Y=out[0])
        call()
        (name, _), = captured_launches(call)
        assert kernel in name
        ref = [o.clone() for o in out]
        for o in out:
            o.fill_(77)
        slow(2_600_000_000)                                       # a wait gives up after 2 s
        call()
        torch.cuda.synchronize()
        assert torq.torq_last_device_error() == 0, kernel
        assert all(torch.equal(o, r) for o, r in zip(out, ref)), kernel
