"""GPU parity of the few-token kernels (rotation up to 256 tokens, GEMM up to 128; the regime where the layer
streams R_inter and W from HBM once): the rotation that splits its contraction over a cluster and reduces the
partial sums through distributed shared memory, and the GEMM built the same way, against the oracle.
Same bounds as everywhere else: rotate + quantize at most 1e-4 of the elements one lattice step off
and 1e-4 of the block scales one step off (one element / block at sizes where 1e-4 is less than
one); GEMM <= 1e-5 relative Frobenius error in fp32, bit-exact where fp32 accumulation is exact."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import captured_launches, dev_bf16, dev_u8, gpu_quantized_to_numpy, lattice, mismatch_report
from paper_2605_19561_b200 import inputs as I
from paper_2605_19561_b200 import torq
import test_gpu_mxint4 as TI
import test_gpu_nvfp4 as TN

pytestmark = pytest.mark.gpu


def _rand_rotation(d, seed):
    """Any well-scaled matrix serves parity (orthogonality is not used by the path); QR only when cheap."""
    g = np.random.default_rng(seed)
    if d <= 1024:
        return I.to_bf16_bits(I.orthogonal(d, g))
    return I.to_bf16_bits(g.standard_normal((d, d)) / np.sqrt(d))


# cluster sizes reached on 148 SMs: d = 128 -> 1, 256 -> 2, 640 -> 5, 1536 -> 8, 2560 -> 7, 4096 -> 4, 5120 -> 3
@pytest.mark.parametrize("M,d", [(1, 128), (16, 256), (17, 256), (32, 640), (33, 640), (64, 1536), (5, 2560),
                                 (48, 4096), (1, 5120), (64, 5120),
                                 # 128 and 256 tokens per instruction (one CTA per SM), two row tiles of scales
                                 (65, 256), (100, 1536), (128, 640), (129, 256), (200, 5120), (256, 2560), (130, 4096)])
def test_rotation_alone_without_any_workspace(M, d):
    g = np.random.default_rng(1000 * M + d)
    xb = I.to_bf16_bits(g.standard_t(3.0, size=(M, d)))
    rb = _rand_rotation(d, d)
    rib = I.to_bf16_bits(I.orthogonal(32, g, batch=d // 32))
    for intra in (rib, None):
        codes_t = torch.full((M, d // 2), 0xEE, dtype=torch.uint8, device="cuda")
        scales_t = torch.full((torq.torq_scales_bytes(M, d),), 0xEE, dtype=torch.uint8, device="cuda")
        before = torq.torq_launch_count()
        torq.torq_rotate_quantize(dev_bf16(xb), dev_bf16(rb), None if intra is None else dev_bf16(intra),
                                  out_codes=codes_t, out_scales=scales_t)
        torch.cuda.synchronize()
        assert torq.torq_launch_count() - before == 1
        assert torq.torq_last_device_error() == 0
        g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
        o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(O.rotate(xb, rb, intra)))
        rep = mismatch_report(g_codes, g_sb, o_codes, o_sb)
        assert rep["non_adjacent"] == 0 and rep["scale_off_by_more_than_one"] == 0, rep
        assert rep["elem_mismatch_frac"] <= max(1e-4, 33.0 / g_codes.size), rep
        assert rep["block_scale_mismatch_frac"] <= max(1e-4, 1.5 / g_sb.size), rep
        # every byte of the scale buffer was written: real rows hold scales, padding rows zero
        raw = scales_t.cpu().numpy().copy()
        rr, cc = np.meshgrid(np.arange(M), np.arange(d // 32), indexing="ij")
        raw[O.scale_layout_offset(rr, cc, d)] = 0
        assert not raw.any()


# the ends of the cluster rule: one K step per CTA (d = 256: four CTAs), more CTAs than SMs (d = 7168: 224),
# 16 feature tiles with one CTA per SM (clusters of 8 would not all fit)
@pytest.mark.parametrize("M,d", [(1, 256), (50, 256), (256, 256), (50, 7168), (100, 2048), (200, 2048)])
def test_rotation_cluster_sizes(M, d):
    test_rotation_alone_without_any_workspace(M, d)


# tokens per instruction go in steps of 16: first and last count of some steps, on both sides of the one-group (pushed)
# form, of one CTA per SM (65) and of the second scale tile (129); one, several and eight CTAs per cluster
@pytest.mark.parametrize("M,d", [(7, 640), (15, 1536), (16, 2560), (17, 896), (48, 896), (49, 1536), (80, 2560), (81, 3072),
                                 (112, 4096), (144, 2176), (145, 4096), (208, 3072), (241, 2176), (12, 12288)])
def test_rotation_token_steps(M, d):
    test_rotation_alone_without_any_workspace(M, d)


# 17 to 32 tokens on clusters that give every group of 8 a CTA of its own, and sizes on the other side of that rule
@pytest.mark.parametrize("M,d", [(17, 1536), (24, 4096), (25, 4096), (33, 2560), (40, 1536), (41, 1536), (18, 256)])
def test_rotation_token_groups_of_eight(M, d):
    test_rotation_alone_without_any_workspace(M, d)
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    P = np.zeros((d, d))
    P[np.arange(d), g.permutation(d)] = 1.0
    pb = I.to_bf16_bits(P)
    TN._rotate_case(xb, pb, None, exact=True)
    TI._rotate_case(xb, pb, None, exact=True)


# 65 to 128 tokens on long K ranges: three stages and two CTAs per SM; d = 5120 and 64 tokens stay as they were
@pytest.mark.parametrize("M,d", [(65, 6400), (128, 6272), (100, 9600)])
def test_rotation_two_ctas_share_an_sm(M, d):
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.standard_t(3.0, size=(M, d)))
    perm = g.permutation(d)                                  # a rotation by one element of each row: sums of one product
    R = torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
    R[torch.arange(d), torch.from_numpy(perm)] = 1.0
    ri = I.to_bf16_bits(I.orthogonal(32, g, batch=d // 32))
    x = dev_bf16(xb)
    for intra in (None, dev_bf16(ri)):
        codes, scales = torq.torq_rotate_quantize(x, R, intra)
        xp = torch.empty_like(x)
        xp[:, torch.from_numpy(perm)] = x
        y = xp.float() if intra is None else torch.einsum("mbk,bkj->mbj", xp.double().view(M, d // 32, 32), intra.double()).reshape(M, d).float()
        torch.cuda.synchronize()
        assert torq.torq_last_device_error() == 0
        g_codes, g_sb = gpu_quantized_to_numpy(codes, scales, M, d)
        o_codes, o_sb = O.quantize_mxfp4(y.cpu().numpy())
        rep = mismatch_report(g_codes, g_sb, o_codes, o_sb)
        assert rep["non_adjacent"] == 0 and rep["elem_mismatch_frac"] <= (0 if intra is None else 1e-4), rep
    # dense: the sum over K, against double precision
    R = (torch.randn(d, d, generator=torch.Generator(device="cuda").manual_seed(d), device="cuda") / d ** 0.5).to(torch.bfloat16)
    y = (x.double() @ R.double()).float()
    codes, scales = torq.torq_rotate_quantize(x, R, None)
    torch.cuda.synchronize()
    rep = mismatch_report(*gpu_quantized_to_numpy(codes, scales, M, d), *O.quantize_mxfp4(y.cpu().numpy()))
    assert rep["non_adjacent"] == 0 and rep["elem_mismatch_frac"] <= 1e-4 and rep["block_scale_mismatch_frac"] <= 1e-4, rep


@pytest.mark.parametrize("M,d", [(65, 6400), (128, 6272)])
def test_rotation_two_ctas_share_an_sm_in_the_other_formats(M, d):
    """The three-stage instances of NVFP4 and MXINT4: permutations of small integers, every code and scale byte exactly."""
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    perm = g.permutation(d)
    R = torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
    R[torch.arange(d), torch.from_numpy(perm)] = 1.0
    y = np.empty((M, d))
    y[:, perm] = O.decode_bf16(xb)
    X = dev_bf16(xb)
    for width in (None, 16, 32):                             # no rotation inside the blocks, a permutation of each
        z, Ri = y, None
        if width is not None:
            pin = np.stack([np.eye(width)[g.permutation(width)] for _ in range(d // width)])
            z = np.einsum("mbk,bkj->mbj", y.reshape(M, d // width, width), pin).reshape(M, d)
            Ri = dev_bf16(I.to_bf16_bits(pin))
            Ri = torq.torq_expand_intra16(Ri) if width == 16 else Ri
        if width != 32:
            ts = O.tensor_scale_from_amax(np.abs(z).max())
            call = lambda: torq.torq_rotate_quantize_nvfp4(X, R, Ri, float(ts))
            g_codes, g_sb = TN._to_numpy(*call(), M, d)
            o_codes, o_sb = O.quantize_nvfp4(z.astype(np.float32), ts)
            assert np.array_equal(g_sb, o_sb) and np.array_equal(g_codes, o_codes)
            assert "ILi1ELi1ELb0ELi3E" in captured_launches(call)[0][0]
        if width != 16:
            call = lambda: torq.torq_rotate_quantize_mxint4(X, R, Ri)
            byt, s = call()
            torch.cuda.synchronize()
            o_q, o_sb = O.quantize_mxint4(z.astype(np.float32))
            assert np.array_equal(TI._operand_to_int(byt), o_q) and np.array_equal(O.unswizzle_scales(s.cpu().numpy(), M, d), o_sb)
            assert "ILi2ELi1ELb0ELi3E" in captured_launches(call)[0][0]
    assert torq.torq_last_device_error() == 0


def test_rotation_exact_cases_are_bit_exact():
    """Permutation and identity rotations with integer activations: every partial sum is exact in any
    order, so codes and scales must equal the oracle's bit for bit through the split and the reduction."""
    d, M = 1536, 40
    g = np.random.default_rng(7)
    x = g.integers(-8, 9, size=(M, d)).astype(np.float64)
    xb = I.to_bf16_bits(x)
    perm = g.permutation(d)
    P = np.zeros((d, d))
    P[np.arange(d), perm] = 1.0
    pin = np.stack([np.eye(32)[g.permutation(32)] for _ in range(d // 32)])
    for rb, rib in ((I.to_bf16_bits(P), I.to_bf16_bits(pin)), (I.to_bf16_bits(np.eye(d)), None)):
        codes_t, scales_t = torq.torq_rotate_quantize(dev_bf16(xb), dev_bf16(rb), None if rib is None else dev_bf16(rib))
        torch.cuda.synchronize()
        g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
        o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(O.rotate(xb, rb, rib)))
        assert np.array_equal(g_sb, o_sb) and np.array_equal(g_codes, o_codes)
    assert torq.torq_last_device_error() == 0


# ------------------------------------------------------------------------------------- GEMM
def _rand_operand(rows, k, seed, scale_lo=118, scale_hi=134):
    g = np.random.default_rng(seed)
    codes = g.integers(0, 16, size=(rows, k), dtype=np.uint8)
    sb = g.integers(scale_lo, scale_hi, size=(rows, k // 32), dtype=np.uint8)
    return codes, sb


def _gpu_gemm(ac, asb, wc, wsb, out_dtype):
    K = ac.shape[1]
    before = torq.torq_launch_count()
    y = torq.torq_mxfp4_gemm(dev_u8(O.pack_codes(ac)), dev_u8(O.swizzle_scales(asb, K, fill=0)),
                             dev_u8(O.pack_codes(wc)), dev_u8(O.swizzle_scales(wsb, K, fill=0)), out_dtype=out_dtype)
    torch.cuda.synchronize()
    assert torq.torq_launch_count() - before == 1
    assert torq.torq_last_device_error() == 0
    return y.float().cpu().numpy().astype(np.float64)


# K = 128 (one half stage), 384 (a half last stage), 640 and 5120 (several stages per split); N ragged in the
# last 128-row tile; cluster sizes 1 .. 8
@pytest.mark.parametrize("M,N,K", [(1, 8, 128), (16, 136, 384), (17, 640, 640), (33, 2560, 1024), (64, 5120, 5120),
                                   (5, 4096, 4096), (64, 264, 2048), (40, 1000, 896),
                                   (65, 136, 384), (100, 2560, 1024), (128, 5120, 5120), (97, 1000, 896)])
def test_gemm_random_operands(M, N, K):
    ac, asb = _rand_operand(M, K, 1)
    wc, wsb = _rand_operand(N, K, 2)
    ref = O.gemm_dequant(ac, asb, wc, wsb)
    got = _gpu_gemm(ac, asb, wc, wsb, torch.float32)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
    # bf16 output: the same fp32 sums, rounded once to nearest even
    gotb = _gpu_gemm(ac, asb, wc, wsb, torch.bfloat16)
    assert np.array_equal(gotb, O.round_to_bf16(got))
    refb = O.round_to_bf16(ref)
    assert np.linalg.norm(gotb - refb) / np.linalg.norm(refb) <= 1e-3


# the ends of the cluster rule: 96 tiles x 2 CTAs, ranges of one and of seven K steps, clusters of eight
@pytest.mark.parametrize("M,N,K", [(33, 12288, 1024), (3, 264, 256), (64, 1024, 14336), (100, 1024, 14336), (100, 2048, 4096)])
def test_gemm_cluster_sizes(M, N, K):
    test_gemm_random_operands(M, N, K)


# the same for the GEMM; K = 256 and 128: a cluster of one CTA, whose accumulator goes to Y directly
@pytest.mark.parametrize("M,N,K", [(3, 1000, 2048), (13, 520, 4096), (16, 264, 384), (48, 1000, 2048), (49, 264, 4096),
                                   (81, 520, 2048), (112, 264, 640), (40, 264, 256), (128, 72, 128), (5, 72, 256)])
def test_gemm_token_steps(M, N, K):
    test_gemm_random_operands(M, N, K)


# more 128-feature tiles than CTAs that fit (one per SM above 64 tokens, two up to there), and the last sizes that fit
@pytest.mark.parametrize("M,N,K", [(65, 18952, 384), (65, 18944, 384), (128, 20480, 256), (100, 28424, 640), (64, 37896, 256),
                                   (49, 37896, 384), (48, 37896, 256)])
def test_gemm_more_tiles_than_fit_at_once(M, N, K):
    test_gemm_random_operands(M, N, K)


def test_gemm_exact_integer_regime_and_one_hot_rows():
    """Equal scales: fp32 accumulation is exact in any order and through the split, so the result is the
    oracle's bit for bit.  One-hot activation rows return single dequantized weight columns: a mix-up of
    row <-> scale or K-block <-> scale on either (swapped) side would show exactly."""
    M, N, K = 48, 400, 1536
    ac, _ = _rand_operand(M, K, 3)
    wc, _ = _rand_operand(N, K, 4)
    asb = np.full((M, K // 32), 127, np.uint8)
    wsb = np.full((N, K // 32), 127, np.uint8)
    assert (_gpu_gemm(ac, asb, wc, wsb, torch.float32) == O.gemm_dequant(ac, asb, wc, wsb)).all()
    g = np.random.default_rng(9)
    wc, wsb = _rand_operand(N, K, 5)
    ac = np.zeros((M, K), np.uint8)
    asb = g.integers(120, 131, size=(M, K // 32), dtype=np.uint8)
    hot = g.integers(0, K, size=M)
    ac[np.arange(M), hot] = 2                              # codeword 1.0
    ref = O.gemm_dequant(ac, asb, wc, wsb)
    assert (_gpu_gemm(ac, asb, wc, wsb, torch.float32) == ref).all()


def test_gemm_leaves_the_neighbours_of_its_output_alone():
    M, N, K = 20, 72, 256
    ac, asb = _rand_operand(M, K, 11)
    wc, wsb = _rand_operand(N, K, 12)
    buf = torch.full((M + 2, N), 777.0, dtype=torch.float32, device="cuda")
    Y = buf[1:M + 1]
    torq.torq_mxfp4_gemm(dev_u8(O.pack_codes(ac)), dev_u8(O.swizzle_scales(asb, K, fill=0)), dev_u8(O.pack_codes(wc)),
                         dev_u8(O.swizzle_scales(wsb, K, fill=0)), Y=Y)
    torch.cuda.synchronize()
    assert bool((buf[0] == 777.0).all()) and bool((buf[M + 1] == 777.0).all())
    ref = O.gemm_dequant(ac, asb, wc, wsb)
    assert np.linalg.norm(Y.cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-5


# K ranges of two steps: the first and last token counts, and sizes on both sides of the line (32 tokens of partial sums per SM)
@pytest.mark.parametrize("M,N,K,ctas", [(17, 256, 4096, 16), (128, 256, 4096, 16), (40, 512, 4096, 32), (64, 1024, 4096, 64), (32, 2048, 4096, 128),
                                        (48, 2048, 4096, 64), (1, 256, 4096, 16), (16, 1024, 4096, 64), (16, 1032, 4096, 72), (16, 2048, 4096, 64),
                                        (24, 520, 3968, 40)])
def test_gemm_few_tiles_split_a_short_contraction_further(M, N, K, ctas):
    ac, asb = _rand_operand(M, K, 1)
    wc, wsb = _rand_operand(N, K, 2)
    ops = (dev_u8(O.pack_codes(ac)), dev_u8(O.swizzle_scales(asb, K, fill=0)), dev_u8(O.pack_codes(wc)), dev_u8(O.swizzle_scales(wsb, K, fill=0)))
    got = torq.torq_mxfp4_gemm(*ops, out_dtype=torch.float32).cpu().numpy()
    ref = O.gemm_dequant(ac, asb, wc, wsb)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        (name, grid), = captured_launches(lambda: torq.torq_mxfp4_gemm(*ops, out_dtype=torch.float32))
        assert "gemm_fewtok_kernel" in name and grid == ctas


# 48 and 58 K steps: clusters of 5 and 6 from 17 to 64 tokens, 4 (5) below and above
@pytest.mark.parametrize("M,d,ctas", [(16, 3072, 96), (17, 3072, 120), (64, 3072, 120), (65, 3072, 96), (33, 3712, 174), (64, 2944, 92)])
def test_rotation_cluster_of_a_contraction_that_just_misses_a_split(M, d, ctas):
    test_rotation_alone_without_any_workspace(M, d)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        X, R = torch.zeros((M, d), dtype=torch.bfloat16, device="cuda"), torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
        (name, grid), = captured_launches(lambda: torq.torq_rotate_quantize(X, R, None))
        assert "rotate_fewtok_kernel" in name and grid == ctas


# tiles that nearly fill the device with clusters of 5 (taken as clusters of 4) and of 3 (whose CTAs leave together up to 128 tokens)
@pytest.mark.parametrize("M,d", [(65, 3200), (128, 3328), (160, 3328), (96, 3072), (65, 5632), (128, 5760), (100, 5760), (160, 5632), (96, 5504)])
def test_rotation_with_clusters_that_nearly_fill_the_device(M, d):
    """Permutations of small integers: every code and scale exactly, three calls in a row on the same buffers."""
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    perm = g.permutation(d)
    P = torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
    P[torch.arange(d, device="cuda"), torch.from_numpy(perm).cuda()] = 1
    pin = np.stack([np.eye(32)[g.permutation(32)] for _ in range(d // 32)])
    y = np.empty((M, d))
    y[:, perm] = O.decode_bf16(xb)
    z = np.einsum("mbk,bkj->mbj", y.reshape(M, d // 32, 32), pin).reshape(M, d)
    X, Ri = dev_bf16(xb), dev_bf16(I.to_bf16_bits(pin))
    codes_t = torch.full((M, d // 2), 0xEE, dtype=torch.uint8, device="cuda")
    scales_t = torch.full((torq.torq_scales_bytes(M, d),), 0xEE, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        torq.torq_rotate_quantize(X, P, Ri, out_codes=codes_t, out_scales=scales_t)
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0
    g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
    o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(z))
    assert np.array_equal(g_sb, o_sb) and np.array_equal(g_codes, o_codes)
    if d in (3200, 3328):
        (name, grid), = captured_launches(lambda: torq.torq_rotate_quantize(X, P, Ri))
        assert "fewtok" not in name or grid == 4 * (d // 128)


# 65 to 80 tokens of byte operands: two sets of epilogue warps where one CTA per SM splits K as far as two would, one set beyond
@pytest.mark.parametrize("M,N,K,sets", [(65, 768, 3072, 2), (80, 1536, 3072, 2), (72, 264, 640, 2), (80, 2560, 3072, 1), (65, 6144, 512, 1), (81, 2560, 3072, 2)])
def test_gemm_mxint4_shares_an_sm_only_for_more_splits(M, N, K, sets):
    aq, asb = TI._rand_operand(M, K, 3)
    wq, wsb = TI._rand_operand(N, K, 4)
    got = TI._gpu_gemm(aq, asb, wq, wsb, torch.float32)
    ref = O.gemm_mxint4(aq, asb, wq, wsb)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        A, W = torch.zeros((M, K), dtype=torch.uint8, device="cuda"), torch.zeros((N, K), dtype=torch.uint8, device="cuda")
        As, Ws = (torch.zeros(torq.torq_scales_bytes(r, K), dtype=torch.uint8, device="cuda") for r in (M, N))
        (name, _), = captured_launches(lambda: torq.torq_mxint4_gemm(A, As, W, Ws))
        assert "wide" in name or f"gemm_fewtok_kernelILi2ELi{sets}E" in name, name


# 65 to 96 tokens: clusters of six from 24 K steps on and up to the tiles that fit; 64 and 97 tokens and 23 tiles as before
@pytest.mark.parametrize("M,d,ctas", [(65, 1536, 72), (96, 1536, 72), (80, 2816, 132), (96, 2304, 108), (64, 1536, 48), (97, 2560, 80), (96, 2944, 92)])
def test_rotation_cluster_with_one_unit_per_cta(M, d, ctas):
    test_rotation_alone_without_any_workspace(M, d)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        X, R = torch.zeros((M, d), dtype=torch.bfloat16, device="cuda"), torch.zeros((d, d), dtype=torch.bfloat16, device="cuda")
        (name, grid), = captured_launches(lambda: torq.torq_rotate_quantize(X, R, None))
        assert "rotate_fewtok_kernel" in name and grid == ctas
