"""Few-token kernels whose partial sums are pushed in pieces of 32 features x 4 tokens (up to 32 tokens, the rotation with R_intra up to 56; the NVFP4 GEMM up to 24): token
counts on both sides of every four, clusters of one CTA to eight, one and several pieces per warp.  Operands whose sums are exact in any
order, so codes, scale bytes, padding and results must equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import captured_launches, dev_bf16, dev_u8, gpu_quantized_to_numpy
from paper_2605_19561_b200 import inputs as I
from paper_2605_19561_b200 import torq
import test_gpu_fewtok as TF
import test_gpu_mxint4 as TI
import test_gpu_nvfp4 as TN

pytestmark = pytest.mark.gpu
E2M1 = np.array([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6])


@pytest.mark.parametrize("M,d", [(1, 128), (2, 256), (3, 19072), (4, 640), (5, 1536), (7, 2560), (8, 5120), (9, 4096), (12, 7168), (13, 9600),
                                 (16, 2048), (17, 128), (20, 14336), (21, 1536), (24, 4096), (28, 2560), (29, 896), (31, 640), (32, 5120),
                                 (30, 19072),
                                 # three stages: 33 to 56 tokens in clusters of eight
                                 (33, 1024), (36, 2048), (37, 3968), (45, 1536), (48, 2432), (49, 2560), (53, 3712), (56, 3072)])
def test_rotation_of_permutations_in_the_three_formats(M, d):
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    perm = g.permutation(d)
    P = torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
    P[torch.arange(d, device="cuda"), torch.from_numpy(perm).cuda()] = 1
    y = np.empty((M, d))
    y[:, perm] = O.decode_bf16(xb)
    X = dev_bf16(xb)
    for width in (None, 16, 32):                             # no rotation inside the blocks, a permutation of each
        z, Ri = y, None
        if width is not None:
            pin = np.stack([np.eye(width)[g.permutation(width)] for _ in range(d // width)])
            z = np.einsum("mbk,bkj->mbj", y.reshape(M, d // width, width), pin).reshape(M, d)
            Ri = dev_bf16(I.to_bf16_bits(pin))
        z = z.astype(np.float32)
        if width != 16:
            codes = torch.full((M, d // 2), 0xEE, dtype=torch.uint8, device="cuda")
            scales = torch.full((torq.torq_scales_bytes(M, d),), 0xEE, dtype=torch.uint8, device="cuda")
            call = lambda: torq.torq_rotate_quantize(X, P, Ri, out_codes=codes, out_scales=scales)
            call()
            torch.cuda.synchronize()
            o_codes, o_sb = O.quantize_mxfp4(z)
            g_codes, g_sb = gpu_quantized_to_numpy(codes, scales, M, d)
            assert np.array_equal(g_codes, o_codes) and np.array_equal(g_sb, o_sb)
            assert np.array_equal(scales.cpu().numpy(), O.swizzle_scales(o_sb, d, fill=0))       # padding rows hold zero
            assert d < 1536 or f"rotate_fewtok_kernelILi0ELi1ELb{int(M <= 32 or width is not None)}E" in captured_launches(call)[0][0]
            byt, s = torq.torq_rotate_quantize_mxint4(X, P, Ri)
            torch.cuda.synchronize()
            o_q, o_sb = O.quantize_mxint4(z)
            assert np.array_equal(TI._operand_to_int(byt), o_q) and np.array_equal(O.unswizzle_scales(s.cpu().numpy(), M, d), o_sb)
        if width != 32:
            ts = O.tensor_scale_from_amax(np.abs(z).max())
            Ri32 = None if Ri is None else torq.torq_expand_intra16(Ri)
            n_codes, n_sb = TN._to_numpy(*torq.torq_rotate_quantize_nvfp4(X, P, Ri32, float(ts)), M, d)
            o_codes, o_sb = O.quantize_nvfp4(z, ts)
            assert np.array_equal(n_sb, o_sb) and np.array_equal(n_codes, o_codes)
    assert torq.torq_last_device_error() == 0


def test_rotation_keeps_what_is_not_a_number_in_its_token():
    """One infinity and one NaN in X reach the outputs of their token only."""
    M, d = 6, 256
    x = np.ones((M, d))
    X = dev_bf16(I.to_bf16_bits(x))
    X[1, 5], X[4, 40] = float("inf"), float("nan")
    E = torch.eye(d, dtype=torch.bfloat16, device="cuda")
    clean, clean_s = torq.torq_rotate_quantize(dev_bf16(I.to_bf16_bits(x)), E, None)
    codes, scales = torq.torq_rotate_quantize(X, E, None)
    torch.cuda.synchronize()
    same = [m for m in range(M) if m not in (1, 4)]
    assert torch.equal(codes.view(M, -1)[same], clean.view(M, -1)[same])
    a, b = (O.unswizzle_scales(t.cpu().numpy(), M, d) for t in (scales, clean_s))
    assert np.array_equal(a[same], b[same])
    assert torq.torq_last_device_error() == 0


# N ragged in a 32-feature piece and in the tile, a half last stage of K, clusters of one to eight
@pytest.mark.parametrize("M,N,K", [(1, 8, 128), (2, 72, 256), (3, 136, 640), (4, 264, 2048), (5, 1000, 2048), (8, 5120, 5120), (9, 520, 4096), (13, 1024, 4096),
                                   (16, 6144, 896), (17, 264, 384), (20, 2560, 1024), (21, 1032, 4096), (24, 4096, 2048), (25, 264, 2048), (29, 72, 4096),
                                   (32, 5120, 1152)])
def test_gemm_of_exact_sums_in_the_three_formats(M, N, K):
    g = np.random.default_rng(M + N + K)
    ac, _ = TF._rand_operand(M, K, 3)
    wc, _ = TF._rand_operand(N, K, 4)
    one = lambda r: np.full((r, K // 32), 127, np.uint8)
    assert (TF._gpu_gemm(ac, one(M), wc, one(N), torch.float32) == O.gemm_dequant(ac, one(M), wc, one(N))).all()
    asb, wsb = (g.choice(np.array([0x30, 0x38, 0x40], np.uint8), size=(r, K // 16)) for r in (M, N))
    got = TN._gpu_gemm(ac, asb, 0.25, wc, wsb, 2.0, torch.float32)
    assert (got == O.gemm_nvfp4(ac, asb, 0.25, wc, wsb, 2.0)).all()      # multiples of 2^-4 up to 36 x 4 K: below 2^24 units
    aq, wq = (g.integers(-7, 8, size=(r, K)).astype(np.int8) for r in (M, N))
    assert (TI._gpu_gemm(aq, one(M), wq, one(N), torch.float32) == O.gemm_mxint4(aq, one(M), wq, one(N))).all()


# Above 16 tokens sums are pushed from K > 2048 on, up to 32 tokens, NVFP4 24: both sides of each line, for a few tiles (clusters of eight)
# and for many (one to four CTAs, so several pieces per warp and both reads of the accumulator).
@pytest.mark.parametrize("M,N,K", [(17, 264, 4096), (20, 1032, 2176), (24, 264, 4096), (25, 520, 2176), (28, 264, 4096), (32, 264, 2176),
                                   (17, 6144, 4096), (20, 6152, 2176), (24, 6144, 4096), (25, 6144, 4096), (28, 5128, 5120), (32, 6144, 4096),
                                   (17, 20480, 2176), (24, 20480, 2176), (32, 20488, 2176), (32, 6144, 2048), (17, 264, 2048), (33, 6144, 4096)])
def test_gemm_of_17_to_32_tokens_on_both_sides_of_the_line(M, N, K):
    g = np.random.default_rng(M + N + K)
    s32 = lambda r: dev_u8(O.swizzle_scales(np.full((r, K // 32), 127, np.uint8), K, fill=0))

    def check(fmt, most, call, ref):
        y = call()
        (name, _), = captured_launches(call)
        assert f"gemm_fewtok_kernelILi{fmt}ELi1ELb{int(M <= most and K > 2048)}E" in name, name
        assert np.array_equal(y.cpu().numpy(), ref.astype(np.float32)), name

    ac, wc = g.integers(0, 16, (M, K), dtype=np.uint8), g.integers(0, 16, (N, K), dtype=np.uint8)
    a, w = dev_u8(O.pack_codes(ac)), dev_u8(O.pack_codes(wc))
    av, wv = E2M1[ac], E2M1[wc]
    ops = (a, s32(M), w, s32(N))
    check(0, 32, lambda: torq.torq_mxfp4_gemm(*ops, out_dtype=torch.float32), av.astype(np.float64) @ wv.T)      # multiples of 1/4 up to 36 K
    asb, wsb = (g.integers(0, 2, (r, K // 16), dtype=np.uint8) for r in (M, N))                                    # E4M3 1 and 2
    opn = (a, dev_u8(O.nv_swizzle_scales((0x38 + 8 * asb).astype(np.uint8), K)), 1.0, w, dev_u8(O.nv_swizzle_scales((0x38 + 8 * wsb).astype(np.uint8), K)), 1.0)
    scaled = lambda v, sb: v * np.repeat(1.0 + sb, 16, axis=1)
    check(1, 24, lambda: torq.torq_nvfp4_gemm(*opn, out_dtype=torch.float32), scaled(av, asb) @ scaled(wv, wsb).T)  # up to 144 K
    ai, wi = (g.integers(-7, 8, (r, K)).astype(np.int8) for r in (M, N))
    opi = (dev_u8(O.int4_to_e4m3(ai)), s32(M), dev_u8(O.int4_to_e4m3(wi)), s32(N))
    check(2, 32, lambda: torq.torq_mxint4_gemm(*opi, out_dtype=torch.float32), ai.astype(np.float64) @ wi.T.astype(np.float64))
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("M,d,kernel", [(6, 2048, "rotate_fewtok_kernelILi0ELi1ELb1ELi5E"), (30, 2560, "rotate_fewtok_kernelILi0ELi1ELb1ELi4E"),
                                        (50, 2560, "rotate_fewtok_kernelILi0ELi1ELb1ELi3E"), (100, 2304, "rotate_fewtok_kernelILi0ELi2ELb0ELi4E"),
                                        (128, 1024, "rotate_quantize_wide_kernelILi0ELi32E"), (300, 2048, "rotate_quantize_wide_kernelILi0ELi128E"),
                                        (1000, 4096, "rotate_quantize_wide_kernelILi0ELi256E"), (1100, 4096, "rotate_quantize_wide_kernelILi0ELi384E"),
                                        (3600, 2048, "rotate_quantize_pair_kernelILi0E")])
def test_every_rotation_keeps_what_is_not_a_number_in_its_token(M, d, kernel):
    """The same with R_intra, through each kernel and each form of the intra rotation: the pieces of the pushed sums, the split terms in
    tensor memory (the one-wave kernel, the pair kernel's last tiles), the warp-level instructions, the FMAs."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the rules are those of 148 SMs")
    g = np.random.default_rng(M)
    x = g.integers(-8, 9, size=(M, d)).astype(np.float64)
    X = dev_bf16(I.to_bf16_bits(x))
    bad = {1, M // 2, M - 2}
    X[1, 5], X[M // 2, d - 40], X[M - 2, d // 2] = float("inf"), float("nan"), float("-inf")
    E = torch.eye(d, dtype=torch.bfloat16, device="cuda")
    Ri = dev_bf16(I.to_bf16_bits(np.stack([np.eye(32)[g.permutation(32)] for _ in range(d // 32)])))
    clean, clean_s = torq.torq_rotate_quantize(dev_bf16(I.to_bf16_bits(x)), E, Ri)
    codes, scales = torq.torq_rotate_quantize(X, E, Ri)
    torch.cuda.synchronize()
    assert kernel in captured_launches(lambda: torq.torq_rotate_quantize(X, E, Ri))[0][0]
    same = torch.tensor([m for m in range(M) if m not in bad], device="cuda")
    assert torch.equal(codes.view(M, -1)[same], clean.view(M, -1)[same])
    a, b = (O.unswizzle_scales(t.cpu().numpy(), M, d)[same.cpu().numpy()] for t in (scales, clean_s))
    assert np.array_equal(a, b)
    assert torq.torq_last_device_error() == 0
