"""GPU parity of the one-wave kernels: the rotation (256 tokens x 32 ... 384 features per CTA pair) on shapes that take it: every
kind of width (one or two instructions, with and without a narrow box, one to three box slots per stage), a ragged
last row tile whose second half has no token, a last column tile that reaches past the last feature, fewer K steps
than pipeline stages; and the GEMM built the same way.  Bounds as in every other parity test."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import captured_launches, dev_bf16, dev_u8, gpu_quantized_to_numpy, mismatch_report
from paper_2605_19561_b200 import inputs as I
from paper_2605_19561_b200 import torq
import test_gpu_mxint4 as TI
import test_gpu_nvfp4 as TN

pytestmark = pytest.mark.gpu


def _rand_rotation(d, seed):
    g = np.random.default_rng(seed)
    return I.to_bf16_bits(g.standard_normal((d, d)) / np.sqrt(d))


# widths on 74 pairs: 32, 32 (two K steps), 32 (padding rows in a second, token-less row tile), 64, 96, 128, 160 (tail of
# 16), 192, 224, 288 (two instructions), 320, 352, 384 (d no multiple of the width but for the first ones)
@pytest.mark.parametrize("M,d", [(50, 256), (24, 128), (16, 256), (1, 128), (257, 256), (700, 1024), (1280, 1024), (1000, 2048), (1280, 2048),
                                 (1536, 2048), (600, 5120), (2304, 2304), (1400, 3840), (3072, 2048), (1280, 5120)])
def test_rotation_mxfp4(M, d):
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.standard_t(3.0, size=(M, d)))
    rb = _rand_rotation(d, d)
    rib = I.to_bf16_bits(I.orthogonal(32, g, batch=d // 32))
    rows = np.unique(np.r_[np.arange(min(M, 64)), np.arange(max(0, M - 140), M), g.integers(0, M, 64)])   # the oracle's share
    for intra in (rib, None):
        codes_t = torch.full((M, d // 2), 0xEE, dtype=torch.uint8, device="cuda")
        scales_t = torch.full((torq.torq_scales_bytes(M, d),), 0xEE, dtype=torch.uint8, device="cuda")
        torq.torq_rotate_quantize(dev_bf16(xb), dev_bf16(rb), None if intra is None else dev_bf16(intra),
                                  out_codes=codes_t, out_scales=scales_t)
        torch.cuda.synchronize()
        assert torq.torq_last_device_error() == 0
        g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
        o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(O.rotate(xb[rows], rb, intra)))
        rep = mismatch_report(g_codes[rows], g_sb[rows], o_codes, o_sb)
        assert rep["non_adjacent"] == 0 and rep["scale_off_by_more_than_one"] == 0, rep
        # one element / block at sizes where 1e-4 is less than one (a block's 32 elements move with its scale)
        assert rep["elem_mismatch_frac"] <= max(1e-4, 33.0 / o_codes.size), rep
        assert rep["block_scale_mismatch_frac"] <= max(1e-4, 1.5 / o_sb.size), rep
        # every byte of the scale buffer was written: real rows hold scales, padding rows zero
        raw = scales_t.cpu().numpy().copy()
        rr, cc = np.meshgrid(np.arange(M), np.arange(d // 32), indexing="ij")
        raw[O.scale_layout_offset(rr, cc, d)] = 0
        assert not raw.any()


def test_rotation_exact_case_is_bit_exact():
    """Permutations of small integers: every partial sum is exact, so codes and scales equal the oracle's bit for bit."""
    M, d = 777, 1280
    g = np.random.default_rng(3)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    P = np.zeros((d, d))
    P[np.arange(d), g.permutation(d)] = 1.0
    pin = I.to_bf16_bits(np.stack([np.eye(32)[g.permutation(32)] for _ in range(d // 32)]))
    codes_t, scales_t = torq.torq_rotate_quantize(dev_bf16(xb), dev_bf16(I.to_bf16_bits(P)), dev_bf16(pin))
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0
    g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
    o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(O.rotate(xb, I.to_bf16_bits(P), pin)))
    assert np.array_equal(g_sb, o_sb) and np.array_equal(g_codes, o_codes)


@pytest.mark.parametrize("M,d", [(600, 1280), (40, 256), (2304, 2304)])
def test_rotation_nvfp4_and_mxint4(M, d):
    cfg = I.CONFIGS["tiny"]
    xb = I.activations(cfg, M=M, d=d)
    rb = _rand_rotation(d, 5)
    TN._rotate_case(xb, rb, I.intra_rotations16(cfg, d=d))
    TN._rotate_case(xb, rb, None)
    g = np.random.default_rng(6)
    TI._rotate_case(xb, rb, I.to_bf16_bits(I.orthogonal(32, g, batch=d // 32)))
    TI._rotate_case(xb, rb, None)


# ------------------------------------------------------------------------------------- GEMM
def _rand_operand(rows, k, seed):
    g = np.random.default_rng(seed)
    return g.integers(0, 16, size=(rows, k), dtype=np.uint8), g.integers(118, 134, size=(rows, k // 32), dtype=np.uint8)


# one-wave GEMM: few tokens with a short contraction; widths 64 and 128 (few output tiles), 192, 320 and 384 (two instructions, W tiles that start 64 rows
# into a scale chunk); ragged rows and columns, a half last K stage (K % 256 == 128)
@pytest.mark.parametrize("M,N,K", [(64, 256, 256), (17, 72, 128), (128, 1032, 512), (1300, 200, 384), (300, 136, 128), (1000, 1000, 256), (2000, 1096, 256), (777, 5120, 2176),
                                   (1000, 6136, 4096)])
def test_gemm_mxfp4(M, N, K):
    ac, asb = _rand_operand(M, K, 1)
    wc, wsb = _rand_operand(N, K, 2)
    ops = (dev_u8(O.pack_codes(ac)), dev_u8(O.swizzle_scales(asb, K, fill=0)), dev_u8(O.pack_codes(wc)),
           dev_u8(O.swizzle_scales(wsb, K, fill=0)))
    rows = np.unique(np.r_[np.arange(min(M, 96)), np.arange(max(0, M - 140), M)])        # the oracle's share
    ref = O.gemm_dequant(ac[rows], asb[rows], wc, wsb)
    out = {}
    for dt in (torch.float32, torch.bfloat16):
        Y = torch.full((M + 2, N), 777.0, dtype=dt, device="cuda")
        torq.torq_mxfp4_gemm(*ops, Y=Y[1:M + 1])
        torch.cuda.synchronize()
        assert torq.torq_last_device_error() == 0
        assert bool((Y[0] == 777).all()) and bool((Y[M + 1] == 777).all())
        out[dt] = Y[1:M + 1].float().cpu().numpy().astype(np.float64)
    got = out[torch.float32][rows]
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.array_equal(out[torch.bfloat16], O.round_to_bf16(out[torch.float32]))     # the same fp32 sums, rounded once


@pytest.mark.parametrize("M,N,K", [(300, 136, 384), (777, 5120, 256)])
def test_gemm_nvfp4_and_mxint4(M, N, K):
    g = np.random.default_rng(3)
    ac, wc = (g.integers(0, 16, (r, K), dtype=np.uint8) for r in (M, N))
    a16, w16 = (g.integers(0x30, 0x40, (r, K // 16), dtype=np.uint8) for r in (M, N))
    y = torq.torq_nvfp4_gemm(dev_u8(O.pack_codes(ac)), dev_u8(O.nv_swizzle_scales(a16, K)), 0.02, dev_u8(O.pack_codes(wc)),
                             dev_u8(O.nv_swizzle_scales(w16, K)), 0.01, out_dtype=torch.float32)
    ref = O.gemm_nvfp4(ac, a16, np.float32(0.02), wc, w16, np.float32(0.01))
    assert np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-5
    aq, wq = (g.integers(-7, 8, (r, K)).astype(np.int8) for r in (M, N))
    asb, wsb = (g.integers(120, 134, (r, K // 32), dtype=np.uint8) for r in (M, N))
    y = torq.torq_mxint4_gemm(dev_u8(O.int4_to_e4m3(aq)), dev_u8(O.swizzle_scales(asb, K, fill=0)), dev_u8(O.int4_to_e4m3(wq)),
                              dev_u8(O.swizzle_scales(wsb, K, fill=0)), out_dtype=torch.float32)
    ref = O.gemm_mxint4(aq, asb, wq, wsb)
    assert np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-5
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("M,d,N", [(257, 256, 256), (441, 256, 1496), (640, 1024, 1024), (257, 256, 248), (640, 1024, 1016), (300, 128, 120),
                                   (641, 512, 504)])
def test_fused_call_of_257_to_640_tokens(M, d, N):
    """The fused call is the separate rotation and GEMM bit for bit, in two launches, whatever N is beside d."""
    g = torch.Generator(device="cuda").manual_seed(M + d + N)
    X = torch.randn(M, d, generator=g, device="cuda").to(torch.bfloat16)
    R = (torch.randn(d, d, generator=g, device="cuda") / d ** 0.5).to(torch.bfloat16)
    Ri = (torch.randn(d // 32, 32, 32, generator=g, device="cuda") / 32 ** 0.5).to(torch.bfloat16)
    Wq = torch.randint(0, 256, (N, d // 2), generator=g, device="cuda", dtype=torch.uint8)
    Ws = torch.randint(120, 132, (torq.torq_scales_bytes(N, d),), generator=g, device="cuda", dtype=torch.uint8)
    codes, scales = torq.torq_rotate_quantize(X, R, Ri)
    ref = torq.torq_mxfp4_gemm(codes, scales, Wq, Ws)
    torch.cuda.synchronize()
    before = torq.torq_launch_count()
    y = torq.torq_rotated_linear(X, R, Ri, Wq, Ws)
    torch.cuda.synchronize()
    assert torq.torq_launch_count() - before == 2
    assert torq.torq_last_device_error() == 0
    assert torch.equal(y, ref)


@pytest.mark.parametrize("M,N,K,kernel", [(129, 8, 128, "wide"), (200, 6144, 4096, "wide"), (256, 9472, 256, "wide"), (256, 128, 14336, "wide"),
                                          (2048, 6144, 4096, "pair"), (100, 28672, 512, "pair")])
def test_gemm_kernel_of_more_than_the_few_tokens(M, N, K, kernel):
    """129 to 256 tokens run on the one-wave kernel however few columns there are; nothing else serves them."""
    A, W = (torch.zeros((r, K // 2), dtype=torch.uint8, device="cuda") for r in (M, N))
    As, Ws = (torch.zeros(torq.torq_scales_bytes(r, K), dtype=torch.uint8, device="cuda") for r in (M, N))
    call = lambda: torq.torq_mxfp4_gemm(A, As, W, Ws)
    y = call()
    (name, _), = captured_launches(call)
    assert f"mxfp4_gemm_{kernel}_kernel" in name and not bool(y.any())
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("M,d", [(40, 384), (128, 896), (130, 128), (300, 640), (300, 1664), (256, 4096)])
def test_rotation_with_two_slabs_per_stage(M, d):
    """Tiles of up to 128 columns, where a stage is 128 of K: one stage, odd numbers of them, more than the ring holds, both
    widths of the last box.  Permutations of small integers: bit for bit the oracle's."""
    g = np.random.default_rng(M + d)
    xb = I.to_bf16_bits(g.integers(-8, 9, size=(M, d)).astype(np.float64))
    P = np.zeros((d, d))
    P[np.arange(d), g.permutation(d)] = 1.0
    pin = I.to_bf16_bits(np.stack([np.eye(32)[g.permutation(32)] for _ in range(d // 32)]))
    rows = np.unique(np.r_[0:min(M, 40), max(0, M - 40):M])
    codes_t, scales_t = torq.torq_rotate_quantize(dev_bf16(xb), dev_bf16(I.to_bf16_bits(P)), dev_bf16(pin))
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0
    g_codes, g_sb = gpu_quantized_to_numpy(codes_t, scales_t, M, d)
    o_codes, o_sb = O.quantize_mxfp4(O.round_to_f32(O.rotate(xb[rows], I.to_bf16_bits(P), pin)))
    assert np.array_equal(g_sb[rows], o_sb) and np.array_equal(g_codes[rows], o_codes)


# tiles of 64 columns on 2, 18 and 33 CTA pairs and of 128 on 24 and 48: four slabs of K, as many as fill one ring (ten), an odd number, a half last
# one, several rounds.  K8: of MXINT4, whose slabs are half as long
@pytest.mark.parametrize("M,N,K,K8", [(200, 72, 1024, 512), (200, 72, 2560, 1280), (300, 520, 1152, 640), (129, 2056, 1280, 640), (513, 1000, 2944, 1408),
                                      (200, 6144, 5376, 2688)])
def test_gemm_with_two_slabs_per_stage(M, N, K, K8):
    """Scales of 1/2, 1 and 2 by row and block and small integers as codes, so that every sum is exact: the three formats equal the product
    bit for bit, and a chunk of scales taken from the other slab of a stage would show.  Each call is of the instance with two slabs."""
    g = np.random.default_rng(M + N + K)
    rows = np.unique(np.r_[0:min(M, 24), max(0, M - 24):M])
    grid = np.array([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6])

    def check(fmt, k, call, av, wv, asb, wsb):
        blk = k // asb.shape[1]
        y = call()
        (name, _), = captured_launches(call)
        assert f"mxfp4_gemm_wide_kernelILi{['mxfp4', 'nvfp4', 'mxint4'].index(fmt)}ELi128E" in name, (fmt, name)
        scaled = lambda v, sb: v * np.repeat(2.0 ** (sb.astype(np.int64) - 1), blk, axis=1)
        assert np.array_equal(y.cpu().numpy()[rows], scaled(av[rows], asb[rows]) @ scaled(wv, wsb).T), fmt

    s32 = lambda sb, k: dev_u8(O.swizzle_scales((126 + sb).astype(np.uint8), k, fill=0))
    s16 = lambda sb, k: dev_u8(O.nv_swizzle_scales((0x30 + 8 * sb).astype(np.uint8), k))                 # E4M3 1/2, 1, 2
    sc = lambda n, k, blk: g.integers(0, 3, (n, k // blk), dtype=np.uint8)
    ac, wc = g.integers(0, 16, (M, K), dtype=np.uint8), g.integers(0, 16, (N, K), dtype=np.uint8)
    a, w = dev_u8(O.pack_codes(ac)), dev_u8(O.pack_codes(wc))
    asb, wsb = sc(M, K, 32), sc(N, K, 32)
    ops = (a, s32(asb, K), w, s32(wsb, K))
    check("mxfp4", K, lambda: torq.torq_mxfp4_gemm(*ops, out_dtype=torch.float32), grid[ac], grid[wc], asb, wsb)
    asb, wsb = sc(M, K, 16), sc(N, K, 16)
    opn = (a, s16(asb, K), 1.0, w, s16(wsb, K), 1.0)
    check("nvfp4", K, lambda: torq.torq_nvfp4_gemm(*opn, out_dtype=torch.float32), grid[ac], grid[wc], asb, wsb)
    ai, wi = g.integers(-7, 8, (M, K8)).astype(np.int8), g.integers(-7, 8, (N, K8)).astype(np.int8)
    asb, wsb = sc(M, K8, 32), sc(N, K8, 32)
    opi = (dev_u8(O.int4_to_e4m3(ai)), s32(asb, K8), dev_u8(O.int4_to_e4m3(wi)), s32(wsb, K8))
    check("mxint4", K8, lambda: torq.torq_mxint4_gemm(*opi, out_dtype=torch.float32), ai.astype(np.float64), wi.astype(np.float64), asb, wsb)
    torch.cuda.synchronize()
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("fmt,M,d,kernel", [("mxfp4", 104, 2048, "wide"), ("mxfp4", 112, 2304, "fewtok"), ("mxfp4", 208, 2816, "wide"),
                                            ("mxint4", 192, 3072, "wide"), ("mxfp4", 192, 4096, "fewtok"), ("mxfp4", 192, 4864, "fewtok"),
                                            ("mxfp4", 216, 4864, "wide"), ("mxfp4", 144, 6912, "wide"), ("nvfp4", 193, 7296, "wide"),
                                            ("mxfp4", 150, 7168, "fewtok"), ("mxint4", 256, 9344, "wide")])
def test_rotation_kernel_of_97_to_256_tokens(fmt, M, d, kernel):
    """The faster of the two kernels on either side of the line, by measurements of both."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is one of 148 SMs")
    X, R = torch.zeros(M, d, dtype=torch.bfloat16, device="cuda"), torch.zeros(d, d, dtype=torch.bfloat16, device="cuda")
    call = {"mxfp4": lambda: torq.torq_rotate_quantize(X, R, None), "nvfp4": lambda: torq.torq_rotate_quantize_nvfp4(X, R, None, 1.0),
            "mxint4": lambda: torq.torq_rotate_quantize_mxint4(X, R, None)}[fmt]
    call()
    (name, _), = captured_launches(call)
    assert {"wide": "rotate_quantize_wide_kernel", "fewtok": "rotate_fewtok_kernel"}[kernel] in name
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("fmt,M,N,K,span", [("mxfp4", 144, 4096, 1152, 256), ("mxfp4", 80, 2048, 1024, 256), ("mxfp4", 144, 512, 1024, 128),
                                            ("mxfp4", 176, 2048, 1280, 256), ("mxfp4", 177, 2048, 1280, 128), ("mxfp4", 144, 4096, 1408, 128),
                                            ("mxfp4", 300, 4096, 768, 256), ("nvfp4", 192, 6144, 1152, 256), ("nvfp4", 192, 6144, 1280, 128),
                                            ("nvfp4", 128, 1536, 1152, 128), ("mxint4", 128, 4096, 512, 256), ("mxint4", 200, 4096, 512, 128),
                                            ("mxint4", 128, 4096, 640, 128), ("mxfp4", 144, 3072, 1280, 128), ("mxfp4", 144, 6144, 1152, 256),
                                            ("mxfp4", 1000, 6144, 4096, 384)])
def test_gemm_takes_two_slabs_per_stage_where_they_are_the_faster(fmt, M, N, K, span):
    """Which instance of the one-wave kernel a call takes, by its template arguments: 128 is the one with two slabs."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is one of 148 SMs")
    A, W = (torch.zeros((r, K if fmt == "mxint4" else K // 2), dtype=torch.uint8, device="cuda") for r in (M, N))
    As, Ws = (torch.zeros(torq.torq_nvfp4_scales_bytes(r, K) if fmt == "nvfp4" else torq.torq_scales_bytes(r, K), dtype=torch.uint8,
                          device="cuda") for r in (M, N))
    call = {"mxfp4": lambda: torq.torq_mxfp4_gemm(A, As, W, Ws), "mxint4": lambda: torq.torq_mxint4_gemm(A, As, W, Ws),
            "nvfp4": lambda: torq.torq_nvfp4_gemm(A, As, 1.0, W, Ws, 1.0)}[fmt]
    call()
    (name, _), = captured_launches(call)
    assert f"mxfp4_gemm_wide_kernelILi{['mxfp4', 'nvfp4', 'mxint4'].index(fmt)}ELi{span}E" in name
    assert torq.torq_last_device_error() == 0


@pytest.mark.parametrize("fmt,M,d", [("mxfp4", 131, 2304), ("mxfp4", 180, 3072), ("mxfp4", 186, 3328), ("mxint4", 205, 3584), ("mxfp4", 225, 3840), ("nvfp4", 245, 4096),
                                     ("mxfp4", 185, 4608), ("mxfp4", 200, 4992), ("mxfp4", 212, 5120), ("mxfp4", 220, 5504), ("mxfp4", 250, 5760)])
def test_rotation_of_129_to_256_tokens_keeps_its_sums_in_parts(fmt, M, d):
    """The few-token kernel contracts K in three to five parts, each in an accumulator of its own, and is the nearer to 64 bits for it: the
    sizes that a line by time alone would give to the kernel with one accumulator."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is one of 148 SMs")
    test_rotation_kernel_of_97_to_256_tokens(fmt, M, d, "fewtok")
