"""The work a program gives this library, as a list of timed cases and a generator of further ones.

Each case names a kind of call and its sizes; `prepare` builds what a program holds before the call (plan, weights, spectra,
workspaces, inputs), `run` makes one pass through the public binding.  Values follow the library's own synthetic workloads
(synth.py): activations ~ N(0,1), long convolution kernels ~ N(0,1) exp(-lam t) / sqrt(n), weights ~ N(0, 1/fan_in).
"""
import math

import torch

from paper_2310_12109_b200 import binding as M

BF16, FP32 = "bf16", "fp32"

# Factorisations of the plan lengths (the tests' and the benchmark's own, and the square ones between them).
DIMS = {256: (16, 16), 512: (32, 16), 1024: (32, 32), 2048: (64, 32), 4096: (64, 64), 8192: (32, 32, 8), 32768: (32, 32, 32)}


def _conv(name, kind, dtype, dims, mode, B, H, n):
    return {**({"name": name} if name else {}), "kind": kind, "dtype": dtype, "dims": "x".join(map(str, dims)), "mode": mode, "B": B, "H": H, "n": n}


def listed():
    return [
        # The smallest call: four short fp32 rows, what a unit test, a probe or a single decode-size request sends.  Latency.
        _conv("conv_fp32_short", "conv", FP32, (32, 16), "causal", 1, 4, 256),
        # The sequence mixer of a BERT-base-shaped encoder at its usual length: 32 sequences of 512, bidirectional.
        _conv("conv_bert_512", "conv", BF16, (32, 16), "circular", 32, 768, 512),
        # The same width at a longer, ragged length, causal: prompts are as long as they are (here 2000 of at most 2048).
        _conv("conv_ragged_2000", "conv", BF16, (64, 64), "causal", 8, 768, 2000),
        # The long causal mixer of a GPT-shaped model: 16384 positions, order-3 plan.
        _conv("conv_gpt_16k", "conv", BF16, (32, 32, 32), "causal", 4, 1024, 16384),
        # One training step's worth of the encoder's mixer: spectrum of the updated kernel, forward, both gradients.
        _conv("conv_train_512", "conv_train", BF16, (32, 16), "circular", 32, 768, 512),
        # The same in fp32 at a medium causal length (order-3 plan of 4096): training where bf16 is not enough.
        _conv("conv_train_fp32_2k", "conv_train", FP32, (16, 16, 16), "causal", 4, 768, 2048),
        # Feature mixing: Monarch matmul of 16384 tokens, 64 blocks of 64 x 64 in both factors.
        {"name": "matmul_16384", "kind": "matmul", "T": 16384},
        # One training step of the same layer on a ragged number of tokens: forward, input gradient, weight gradients.
        {"name": "matmul_train_5001", "kind": "matmul_train", "T": 5001},
        # The M2 operator M_b (K (.) M_a X) of the paper's operator benchmark: N = 64K, 768 columns.
        {"name": "operator_64k", "kind": "operator", "b": 256, "d": 768},
        # Inference through the whole M2 block of the BERT-base shape: gated mixer and block-diagonal MLP.
        {"name": "block_bert", "kind": "block", "B": 32},
        # The causal Hyena layer with heads of 16 (language-model mixer), 32 sequences of 256.
        {"name": "hyena_256", "kind": "hyena", "B": 32, "n": 256, "d": 768},
        # The gated bidirectional mixer with dense projections of M2-BERT, 32 sequences of 512.
        {"name": "bert_mixer", "kind": "mixer", "B": 32, "d": 768},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "conv_train", "conv_train", "matmul", "matmul_train", "operator", "block", "hyena", "mixer"])
    if kind in ("conv", "conv_train"):
        dtype = rng.choice([BF16, BF16, FP32])
        # fp32 rows, and rows of which a gradient is taken, stay at 8192 points; the longest plan is for bf16 inference
        N = rng.choice([n for n in DIMS if n <= 8192 or (kind == "conv" and dtype == BF16)])
        mode = rng.choice(["causal", "circular"])
        # a causal program takes the smallest plan its length fits in; half of the lengths are the full ones
        n = N if mode == "circular" else rng.choice([N // 2, rng.randint(N // 4 + 1, N // 2)])
        H = rng.choice([4, 64, 100, 256, 768, 1024])
        rows = (1 << 24 if kind == "conv" else 1 << 23) // N
        B = _log_int(rng, 1, max(1, min(32, rows // H)))
        return _conv("", kind, dtype, DIMS[N], mode, B, min(H, rows), n)
    if kind == "matmul":
        return {"kind": kind, "T": _log_int(rng, 1, 16384)}
    if kind == "matmul_train":
        return {"kind": kind, "T": _log_int(rng, 16, 5001)}
    if kind == "operator":
        b = rng.choice([64, 128, 256])
        return {"kind": kind, "b": b, "d": 8 * _log_int(rng, 8, 96)}
    if kind == "block":
        return {"kind": kind, "B": rng.randint(1, 32)}
    if kind == "hyena":
        return {"kind": kind, "B": _log_int(rng, 1, 32), "n": 8 * rng.randint(8, 32), "d": 64 * rng.randint(2, 12)}
    return {"kind": "mixer", "B": _log_int(rng, 1, 32), "d": 64 * rng.randint(2, 12)}


class _Draw:
    """Normal tensors on the GPU from one seed."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda").manual_seed(seed)

    def __call__(self, shape, scale=1.0, dtype=torch.float32):
        return (torch.randn(shape, generator=self.gen, device="cuda") * scale).to(dtype)

    def kernel(self, H, n):
        """Long convolution kernels: N(0,1) exp(-lam t) / sqrt(n), fp32; lam as in the short and in the long configuration."""
        lam = (2.56 if n <= 512 else 8.192) / n
        t = torch.arange(n, device="cuda", dtype=torch.float32)
        return (self((H, n)) * torch.exp(-lam * t) / math.sqrt(n)).contiguous()


def _dims(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _plan(dims, dtype):
    return M.Plan(dims, dtype=M.M2_BF16 if dtype == BF16 else M.M2_FP32, device=torch.cuda.current_device())


def prepare(case, seed):
    rnd, kind, bf = _Draw(seed), case["kind"], torch.bfloat16
    s = {"kind": kind}
    if kind in ("conv", "conv_train"):
        tdt = bf if case["dtype"] == BF16 else torch.float32
        B, H, n = case["B"], case["H"], case["n"]
        s["plan"] = plan = _plan(_dims(case), case["dtype"])
        s["mode"] = M.M2_CAUSAL if case["mode"] == "causal" else M.M2_CIRCULAR
        s["x"] = rnd((B, H, n), 1.0, tdt)
        s["k"] = rnd.kernel(H, n)
        if kind == "conv":   # inference: the spectrum is computed once per weight update
            s["kf"] = M.m2_kernel_spectrum(plan, s["k"])
        else:
            s["g"] = rnd((B, H, n), 1.0, tdt)
    elif kind in ("matmul", "matmul_train"):
        T = case["T"]
        s["plan"] = plan = _plan((64, 64), BF16)
        s["X"] = rnd((T, 4096), 1.0, bf)
        s["L"], s["R"] = rnd((64, 64, 64), 1 / 8, bf), rnd((64, 64, 64), 1 / 8, bf)
        s["ws"] = M.m2_matmul_workspace(plan, T)
        if kind == "matmul_train":
            s["G"] = rnd((T, 4096), 1.0, bf)
    elif kind == "operator":
        b, d = case["b"], case["d"]
        s["plan"] = _plan((b, b), BF16)
        s["X"], s["K"] = rnd((1, b * b, d), 1.0, bf), rnd((b * b, d), 1.0, bf)
        s["W"] = [rnd((b, b, b), 1 / math.sqrt(b), bf) for _ in range(4)]
        s["ws"] = torch.empty_like(s["X"])
    elif kind == "block":
        s["plan"] = plan = _plan((32, 16), BF16)
        s["x"] = rnd((case["B"], 512, 768), 1.0, bf)
        s["kf"] = M.m2_kernel_spectrum(plan, rnd.kernel(768, 512))
        s["w"] = rnd((768, 3), 1 / math.sqrt(3))
        s["up"], s["down"] = rnd((4, 768, 192), 1 / math.sqrt(192), bf), rnd((4, 192, 768), 1 / math.sqrt(768), bf)
    elif kind == "hyena":
        B, n, d = case["B"], case["n"], case["d"]
        s["plan"] = plan = _plan((32, 16), BF16)
        s["u"] = rnd((B, n, d), 1.0, bf)
        s["W"] = [rnd((d, d), 1 / math.sqrt(d), bf) for _ in range(4)]
        s["kf"] = [M.m2_kernel_spectrum(plan, rnd.kernel(d, n)) for _ in range(3)] + [M.m2_kernel_spectrum(plan, rnd.kernel(d // 16, n))]
        s["scratch"] = M.m2_hyena_scratch(plan, B, n, d, 16)
    else:
        B, d = case["B"], case["d"]
        s["plan"] = plan = _plan((32, 16), BF16)
        s["x"] = rnd((B, 512, d), 1.0, bf)
        s["W"] = [rnd((d, d), 1 / math.sqrt(d), bf) for _ in range(4)]
        s["w"] = [rnd((d, 3), 1 / math.sqrt(3)) for _ in range(3)]
        s["kf"], s["kf_res"] = M.m2_kernel_spectrum(plan, rnd.kernel(d, 512)), M.m2_kernel_spectrum(plan, rnd.kernel(d, 512))
        s["scratch"] = torch.empty(8 * B * 512 * d * 2, dtype=torch.uint8, device="cuda")   # eight bf16 tensors of x's size
    return s


def run(s):
    plan, kind = s["plan"], s["kind"]
    if kind == "conv":
        return M.m2_monarch_conv_fwd(plan, s["x"], s["kf"], s["mode"])
    if kind == "conv_train":
        kf = M.m2_kernel_spectrum(plan, s["k"])
        y = M.m2_monarch_conv_fwd(plan, s["x"], kf, s["mode"])
        dx = M.m2_monarch_conv_fwd(plan, s["g"], M.m2_spectrum_conjugate(plan, kf, s["k"].shape[0]), s["mode"])
        dk = M.m2_monarch_conv_bwd_kernel(plan, s["x"], s["g"], s["mode"])
        return {"y": y, "dx": dx, "dk": dk}
    if kind == "matmul":
        return M.m2_monarch_matmul(plan, s["X"], s["L"], s["R"], ws=s["ws"])
    if kind == "matmul_train":
        Y = M.m2_monarch_matmul(plan, s["X"], s["L"], s["R"], ws=s["ws"])
        dX = M.m2_monarch_matmul_bwd_input(plan, s["G"], s["L"], s["R"], ws=s["ws"])
        dL, dR = M.m2_monarch_matmul_bwd_weights(plan, s["X"], s["G"], s["L"], s["R"])
        return {"Y": Y, "dX": dX, "dL": dL, "dR": dR}
    if kind == "operator":
        La, Ra, Lb, Rb = s["W"]
        Z = M.m2_monarch_cols(plan, s["X"], La, Ra, K=s["K"], ws=s["ws"])
        return M.m2_monarch_cols(plan, Z, Lb, Rb, ws=s["ws"])
    if kind == "block":
        return M.m2_block_fwd(plan, s["x"], s["kf"], s["w"], s["up"], s["down"])[0]
    if kind == "hyena":
        return M.m2_hyena_heads_fwd(plan, s["u"], s["W"], *s["kf"], 16, scratch=s["scratch"])
    return M.m2_bert_mixer_fwd(plan, s["x"], s["W"], s["w"], s["kf"], s["kf_res"], scratch=s["scratch"])


def _conv_flops(rows, N):
    """One real convolution per row, by a fast transform: two real transforms of N points and half a spectrum of products."""
    return rows * (2 * 2.5 * N * math.log2(N) + 3 * N)


def work(case):
    kind = case["kind"]
    if kind in ("conv", "conv_train"):
        N, es = math.prod(_dims(case)), 2 if case["dtype"] == BF16 else 4
        B, H, n = case["B"], case["H"], case["n"]
        if kind == "conv":     # x and y, and the spectrum of a real kernel (half of it determines the rest)
            return {"bytes": 2 * B * H * n * es + H * N * 4, "flops": _conv_flops(B * H, N)}
        # x, g, k in; y, dx, dk out
        return {"bytes": 4 * B * H * n * es + 2 * H * n * 4, "flops": 2 * _conv_flops(B * H, N)}
    if kind == "matmul":
        return {"bytes": 2 * case["T"] * 4096 * 2 + 2 * 64 ** 3 * 2, "flops": 4 * case["T"] * 4096 * 64}
    if kind == "matmul_train":   # X, G, L, R in; Y, dX (bf16), dL, dR (fp32) out
        return {"bytes": 4 * case["T"] * 4096 * 2 + 2 * 64 ** 3 * (2 + 4), "flops": 3 * 4 * case["T"] * 4096 * 64}
    if kind == "operator":
        b, d = case["b"], case["d"]
        return {"bytes": 3 * b * b * d * 2 + 4 * b ** 3 * 2, "flops": 8 * b ** 3 * d}
    if kind == "block":
        t = case["B"] * 512
        return {"bytes": 2 * t * 768 * 2 + 2 * 4 * 768 * 192 * 2 + 768 * 512 * 4, "flops": 4 * t * 768 * 768 + _conv_flops(case["B"] * 768, 512)}
    if kind == "hyena":   # four projections, three short convolutions; per head scores, their product with the kernel, values
        B, n, d = case["B"], case["n"], case["d"]
        return {"bytes": 2 * B * n * d * 2 + 4 * d * d * 2 + (3 * d + d // 16) * 512 * 4,
                "flops": 8 * B * n * d * d + _conv_flops(3 * B * d, 512) + 2 * B * n * n * d}
    B, d = case["B"], case["d"]
    return {"bytes": 2 * B * 512 * d * 2 + 4 * d * d * 2 + 2 * d * 512 * 4, "flops": 8 * B * 512 * d * d + _conv_flops(2 * B * d, 512)}


def tolerance(case):
    # about four times the distance from the same path in 64 bits: 2e-7 to 3.5e-7 in fp32; 1.7e-3 where a bf16 row is rounded on
    # storage only, up to 5e-3 where the operands of every stage are bf16, 1e-2 for the Hyena layer's seven roundings in a row
    if case.get("dtype") == FP32:
        return {"rel": 1.5e-6}
    if case["kind"] in ("conv", "conv_train") and math.prod(_dims(case)) not in (512, 32768):
        return {"rel": 6e-3}
    if case["kind"] in ("matmul", "matmul_train"):
        return {"rel": 1e-2}
    return {"rel": 3e-2 if case["kind"] == "hyena" else 1.5e-2}
