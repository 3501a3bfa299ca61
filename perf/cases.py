"""Workloads of the rotated 4-bit linear layer, for timing and for comparing two builds of the library.

One case is one call of the whole layer (rotate, quantize, block-scaled GEMM) on M tokens, d input and N
output features, as a serving program makes it: the rotations and the prepared weights are laid out once per
layer, the scratch and the output buffer are kept, the activations are what changes from call to call.
"""
import math

import torch

from paper_2605_19561_b200 import torq

# (d, N, activation distribution, outlier channels, outlier gain) of the layers of inputs.CONFIGS
_LAYERS = {
    "tiny": (256, 256, "student_t3", 4, 50.0),
    "llama3_8b_qkv": (4096, 6144, "student_t3", 4, 100.0),
    "llama3_8b_down": (14336, 4096, "laplace", 8, 200.0),
    "qwen3_32b_gateup": (5120, 51200, "student_t3", 5, 100.0),
    "qwen3_32b_sweep": (5120, 5120, "student_t3", 0, 1.0),
}
_MAX_TOKENS = 16384
_MAX_COST = 8192 * 5120 * (5120 + 51200)         # M d (d + N) of the largest listed case


def _case(layer, M, fmt="mxfp4", out="bf16", merged=False):
    d, N, dist, n_outliers, gain = _LAYERS[layer]
    return {"fmt": fmt, "M": M, "d": d, "N": N, "dist": dist, "outliers": n_outliers, "gain": gain, "out": out,
            "merged": merged}


def listed():
    return [
        # the smallest layer of the test suite, float32 result: launches and latency only
        dict(_case("tiny", 64, out="f32"), name="tiny_fp32"),
        # one sequence being decoded: R_inter and W are streamed once for a single token
        dict(_case("qwen3_32b_sweep", 1), name="decode_1"),
        # a small decode batch in the NVFP4 format
        dict(_case("llama3_8b_qkv", 24, fmt="nvfp4"), name="decode_24_nvfp4"),
        # a larger decode batch on the layer with the largest rotation (411 MB)
        dict(_case("llama3_8b_down", 50), name="decode_50_down"),
        # a short prompt, or a large decode batch
        dict(_case("llama3_8b_qkv", 200), name="prompt_200"),
        # a prompt of ordinary length that is no multiple of any tile
        dict(_case("qwen3_32b_sweep", 777), name="prompt_777"),
        # the two LLaMA3-8B prefill shapes
        dict(_case("llama3_8b_qkv", 2048), name="prefill_qkv"),
        dict(_case("llama3_8b_down", 2048), name="prefill_down"),
        # long prefill through a gate/up projection: the largest call
        dict(_case("qwen3_32b_gateup", 8192), name="prefill_gateup"),
        # ragged prefill in the NVFP4 format
        dict(_case("llama3_8b_qkv", 1900, fmt="nvfp4"), name="prefill_nvfp4"),
        # prefill in the MXINT4 format
        dict(_case("llama3_8b_qkv", 2048, fmt="mxint4"), name="prefill_mxint4"),
        # prefill with the rotation in its Kronecker structure (one matrix across blocks, one inside)
        dict(_case("llama3_8b_qkv", 2048, fmt="structured"), name="prefill_structured"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more layer call: the configured layers or any other sizes between them, 1 to 16384 tokens."""
    fmt = rng.choice(["mxfp4"] * 6 + ["nvfp4"] * 2 + ["mxint4"] + ["structured"] * 2)
    c = _case(rng.choice(sorted(_LAYERS)), 1, fmt)
    if rng.random() < 0.5:                       # sizes of no configured layer
        step = 256 if fmt == "structured" else 128
        c["d"] = step * max(1, _log_int(rng, 256, 14336) // step)
        c["N"] = 8 * _log_int(rng, 32, 2048)
        c["dist"] = rng.choice(["student_t3", "laplace"])
        c["outliers"], c["gain"] = rng.randrange(0, 9), rng.choice([50.0, 100.0, 200.0])
    c["M"] = _log_int(rng, 1, min(_MAX_TOKENS, _MAX_COST // (c["d"] * (c["d"] + c["N"]))))
    c["out"] = "f32" if rng.random() < 0.1 else "bf16"
    c["merged"] = fmt != "structured" and rng.random() < 0.1
    return c


def _gaussian(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _orthogonal(g, n, batch=None):
    q, r = torch.linalg.qr(_gaussian(g, n, n) if batch is None else _gaussian(g, batch, n, n))
    return q * torch.sign(torch.diagonal(r, dim1=-2, dim2=-1)).unsqueeze(-2)


def _dense_orthogonal(g, d):
    """Dense d x d orthogonal matrix (d a multiple of 128) without a d x d factorisation: a Kronecker product of
    two random orthogonal matrices, rows and columns permuted, column signs random."""
    q = torch.kron(_orthogonal(g, d // 128), _orthogonal(g, 128))
    q = q[torch.randperm(d, generator=g, device="cuda")][:, torch.randperm(d, generator=g, device="cuda")]
    return (q * torch.sign(_gaussian(g, d))).to(torch.bfloat16).contiguous()


def _activations(g, case):
    M, d = case["M"], case["d"]
    x = _gaussian(g, M, d)
    if case["dist"] == "student_t3":             # normal over the root of a chi-square with 3 degrees of freedom / 3
        s = torch.zeros_like(x)
        for _ in range(3):
            s += _gaussian(g, M, d).square_()
        x /= s.div_(3.0).sqrt_()
    else:                                        # Laplace(0, 1)
        u = torch.rand(M, d, generator=g, device="cuda").clamp_(1e-7)
        x = torch.sign(x) * -torch.log(u)
    if case["outliers"]:
        x[:, torch.randperm(d, generator=g, device="cuda")[:case["outliers"]]] *= case["gain"]
    return x.to(torch.bfloat16).contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    fmt, M, d, N = case["fmt"], case["M"], case["d"], case["N"]
    s = {"fmt": fmt, "X": _activations(g, case)}
    if fmt == "structured":
        s["R"] = _orthogonal(g, d // 32).to(torch.bfloat16).contiguous()
        s["Ri"] = _orthogonal(g, 32).to(torch.bfloat16).contiguous()
        # the dense pair it stands for: R_inter = R_B^T (x) I_32, the same R_intra in every block
        r_inter = torch.kron(s["R"].t().contiguous(), torch.eye(32, dtype=torch.bfloat16, device="cuda"))
        r_intra = s["Ri"].expand(d // 32, 32, 32).contiguous()
    else:
        r_inter = _dense_orthogonal(g, d)
        if fmt == "nvfp4":
            r_intra = torq.torq_expand_intra16(_orthogonal(g, 16, d // 16).to(torch.bfloat16).contiguous())
        else:
            r_intra = _orthogonal(g, 32, d // 32).to(torch.bfloat16).contiguous()
        if case["merged"]:
            r_inter, r_intra = torq.torq_merge_rotations_bf16(r_inter, r_intra), None
        s["R"], s["Ri"] = r_inter, r_intra
    W = _gaussian(g, d, N) * 0.02
    if fmt == "nvfp4":
        s["Wq"], s["Ws"], s["w_scale"] = torq.torq_prepare_weights_nvfp4(r_inter, r_intra, W)
        s["x_scale"] = float((s["X"] @ r_inter).abs().max()) / (6 * 448)      # calibrated ahead of time
        size = torq.torq_nvfp4_workspace_bytes(M, d, N)
    elif fmt == "mxint4":
        _, s["Wq"], s["Ws"] = torq.torq_prepare_weights_mxint4(r_inter, r_intra, W)
        size = torq.torq_mxint4_workspace_bytes(M, d, N)
    else:
        s["Wq"], s["Ws"] = torq.torq_prepare_weights(r_inter, r_intra, W)
        size = torq.torq_workspace_bytes(M, d, N)
    s["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    s["Y"] = torch.empty((M, N), dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16, device="cuda")
    return s


def run(s):
    if s["fmt"] == "nvfp4":
        return torq.torq_rotated_linear_nvfp4(s["X"], s["R"], s["Ri"], s["x_scale"], s["Wq"], s["Ws"], s["w_scale"],
                                              Y=s["Y"], workspace=s["workspace"])
    layer = {"mxfp4": torq.torq_rotated_linear, "mxint4": torq.torq_rotated_linear_mxint4,
             "structured": torq.torq_rotated_linear_structured}[s["fmt"]]
    return layer(s["X"], s["R"], s["Ri"], s["Wq"], s["Ws"], Y=s["Y"], workspace=s["workspace"])


def work(case):
    M, d, N = case["M"], case["d"], case["N"]
    w_bytes = d * N if case["fmt"] == "mxint4" else d * N // 2
    w_bytes += d * N // (16 if case["fmt"] == "nvfp4" else 32)                # block scales
    if case["fmt"] == "structured":
        r_bytes, r_flops = 2 * (d // 32) ** 2 + 2 * 32 * 32, 2 * M * d * (d // 32 + 32)
    else:
        r_bytes = 2 * d * d + (0 if case["merged"] else 64 * d)
        r_flops = 2 * M * d * (d + (0 if case["merged"] else 32))
    y_bytes = M * N * (4 if case["out"] == "f32" else 2)
    return {"bytes": 2 * M * d + r_bytes + w_bytes + y_bytes, "flops": r_flops + 2 * M * d * N}


def tolerance(case):
    # Against the same path with both rotations and the product in 64 bits the output differs by 1.65e-3 to 3.5e-3
    # (relative 2-norm, growing with d): 1.65e-3 is the rounding to bf16, the rest comes from the few elements per
    # million whose rotated value lies so close to a rounding threshold of the quantizer that the order of the sum
    # decides (up to 3.4e-3 at d = 14336, which a float32 result shows as well).
    return {"rel": 1e-2}
