"""The work this library is used for, as cases of a speed comparison.

A case is one pass through the public binding, with the inputs, the workspace and the gradients a training step has
in hand before the call.  Six kinds of pass:

  step      forward and backward of a linear consumer: ``compress`` of the saved activation, ``weight_grad`` of all its
            LoRA consumers from the factors (bf16 and fp32; power_iters > 0 runs the loop of Algorithm 1)
  prenorm   the pre-norm unit: ``compress_prenorm`` (RMS or LayerNorm) and the weight gradients of its projections;
            for RMS also ``prenorm_backward``
  wgrad     one ``weight_grad`` call on factors that a forward pass left behind
  rebuild   ``reconstruct``: the activation rebuilt from its factors
  act       ``activation_backward``: the gradient through SiLU or GELU at the rebuilt activation

Sizes are those of ``synth.WORKLOADS`` and of its long-context sweep, a ragged shape of the parity tests' kind, and, in
``draw``, sizes between the smallest and the largest of these.
"""
import math

import torch

from paper_2509_23472_b200 import binding, synth

# Spectra of the inputs: those of the workloads in synth (nominal singular values of the signal part).
_SPECTRA = ("exp", "pow1", "pow1.5", "geom")


def _case(name, kind, n, d, r, g, dtype="bf16", pad=0, t=0, norm="", act="", spectrum="exp", signal=0, noise=1e-2):
    c = {"kind": kind, "n": n, "d": d, "r": r, "g": g, "dtype": dtype, "pad": pad, "t": t, "norm": norm, "act": act,
         "spectrum": spectrum, "signal": signal or min(2 * r, 1024), "noise": noise}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the small fp32 configuration: a call of a few hundred rows, all latency
        _case("f32_small_step", "step", 512, 768, 64, 16, dtype="f32", spectrum="geom", signal=48, noise=1e-3),
        # one weight gradient at the backward pass of one LoRA consumer: the smallest call of a training step
        _case("wgrad_one_consumer", "wgrad", 4096, 5120, 64, 16, signal=768),
        # ViT-B/16, 64 images: LayerNorm input shared by the q / k / v adapters
        _case("vit_layernorm_unit", "prenorm", 64 * 197, 768, 96, 48, norm="layer", spectrum="pow1.5", signal=128),
        # long-context sweep, shortest context at the lowest rank
        _case("short_context_r64_step", "step", 4096, 5120, 64, 16, signal=768),
        # a token count, a width and a rank that fill no tile, and a row stride wider than the row
        _case("ragged_step", "step", 5003, 1000, 336, 23, pad=24, spectrum="pow1", signal=700),
        # the loop of Algorithm 1 (one power iteration), for inputs whose outlier tokens a row sample can miss
        _case("power_iteration_step", "step", 8192, 5120, 128, 16, t=1, signal=768),
        # LLaMA pre-norm unit, forward and backward
        _case("rms_unit_forward_backward", "prenorm", 8192, 4096, 128, 96, norm="rms", signal=512),
        # LLaMA-7B block input, six LoRA consumers: the benchmark's step
        _case("llama7b_block_step", "step", 16384, 4096, 256, 96, signal=512),
        # the same activation rebuilt in the backward pass of a consumer that needs it whole
        _case("llama7b_block_rebuild", "rebuild", 16384, 4096, 256, 0, signal=512),
        # the feed-forward activation of LLaMA-7B: gradient through SiLU at the rebuilt input
        _case("llama7b_mlp_silu_backward", "act", 16384, 11008, 512, 0, act="silu", spectrum="pow1", signal=1024),
        # the same activation compressed for down_proj: the widest input
        _case("llama7b_mlp_step", "step", 16384, 11008, 512, 16, spectrum="pow1", signal=1024),
        # long-context sweep, longest context at the highest rank: the largest call, two orthonormalisation rounds
        _case("long_context_r512_step", "step", 32768, 5120, 512, 16, signal=768),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "prenorm", "prenorm", "wgrad", "rebuild", "act"))
    dtype = "f32" if kind in ("step", "wgrad", "rebuild") and rng.random() < 0.2 else "bf16"
    top_n, top_d, top_r = (2048, 2048, 192) if dtype == "f32" else (32768, 11008, 512)
    while True:
        n, d = _log(rng, 384, top_n), _log(rng, 256, top_d) // 8 * 8
        r = _log(rng, 16, top_r) // 16 * 16
        # no more work than the largest listed case, a rank well below both extents (it is a compression), and, for
        # bf16, an input of a size somebody compresses
        if n * d <= 16384 * 11008 // 2 and 2 * r <= min(n, d) and (dtype == "f32" or n * d >= 1 << 19):
            break
    if rng.random() < 0.3:
        n = max(384, n // 128 * 128)        # whole tiles are as common as odd token counts
    norm = rng.choice(("rms", "layer")) if kind == "prenorm" else ""
    return _case("", kind, n, d, r, 0 if kind in ("rebuild", "act") else _log(rng, 8, 128), dtype=dtype,
                 pad=8 * rng.randint(1, 4) if kind == "step" and rng.random() < 0.25 else 0,
                 t=1 if kind == "step" and dtype == "bf16" and rng.random() < 0.2 else 0,
                 norm=norm, act=rng.choice(("silu", "gelu")) if kind == "act" else "",
                 spectrum="geom" if dtype == "f32" else rng.choice(("exp", "pow1", "pow1.5")),
                 signal=min(2 * r, 1024, min(n, d)), noise=1e-3 if dtype == "f32" else 1e-2)


def _sigma(case):
    i = torch.arange(1, case["signal"] + 1, dtype=torch.float64)
    s = {"exp": torch.exp(-i * (12.0 / case["signal"])), "pow1": 1.0 / i, "pow1.5": i ** -1.5,
         "geom": torch.exp(-i * (5.0 / case["signal"]))}[case["spectrum"]]
    return s.to(torch.float32)


def prepare(case, seed):
    """An activation with a long-tailed spectrum (the workloads' recipe), the upstream gradients, a workspace."""
    dev = torch.device("cuda")
    n, d, r, g = case["n"], case["d"], case["r"], case["g"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed + 1000)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev, dtype=torch.float32)

    X = synth.low_rank_plus_noise(n, d, case["signal"], _sigma(case), case["noise"], seed, dtype, dev)
    if case["pad"]:   # a column range of a wider buffer: the row stride exceeds the row
        wide = torch.zeros(n, d + case["pad"], dtype=dtype, device=dev)
        wide[:, :d] = X
        X = wide[:, :d]
    s = {"case": case, "seed": seed, "X": X, "ws": binding.alloc_workspace(binding.make_desc(X, r), dev)}
    if g:
        s["G"] = normal(n, (g + 7) // 8 * 8).to(dtype)[:, :g]
    if case["norm"]:
        s["gamma"] = (1.0 + 0.1 * normal(d)).to(dtype)
        s["beta"] = (0.1 * normal(d)).to(dtype) if case["norm"] == "layer" else None
        if case["norm"] == "rms":
            s["grad_A"] = normal(n, d).to(dtype)
    if case["kind"] in ("wgrad", "rebuild", "act"):
        # factors as a forward pass leaves them behind, made here without the library: an orthonormal basis of the
        # range of X S^T for r rows S of X, and its coefficients
        X32 = s.pop("X").float()
        U = torch.linalg.qr(X32 @ X32[torch.randperm(n, generator=gen, device=dev)[:r]].t())[0].to(dtype)
        s["U"], s["V"] = U.contiguous(), (U.float().t() @ X32).to(dtype).contiguous()
    if case["kind"] == "act":
        s["grad_Z"] = normal(n, d).to(dtype)
    return s


def run(s):
    c, ws = s["case"], s["ws"]
    kind, r = c["kind"], c["r"]
    if kind == "step":
        U, V, idx = binding.compress(s["X"], r, seed=s["seed"], call_id=1, ws=ws, power_iters=c["t"])
        return U, V, idx, binding.weight_grad(U, V, s["G"], ws=ws)
    if kind == "prenorm":
        layer = c["norm"] == "layer"
        A, rstd, mean, U, V, idx = binding.compress_prenorm(
            s["X"], s["gamma"], s["beta"], 1e-5 if layer else 1e-6, binding.NORM_LAYER if layer else binding.NORM_RMS,
            r, seed=s["seed"], call_id=1, ws=ws)
        dW = binding.weight_grad(U, V, s["G"], ws=ws)
        if layer:
            return A, rstd, mean, U, V, idx, dW
        return A, rstd, U, V, idx, dW, binding.prenorm_backward(U, V, s["gamma"], rstd, s["grad_A"], ws=ws)
    if kind == "wgrad":
        return binding.weight_grad(s["U"], s["V"], s["G"], ws=ws)
    if kind == "rebuild":
        return binding.reconstruct(s["U"], s["V"])
    return binding.activation_backward(s["U"], s["V"], s["grad_Z"],
                                       binding.ACT_SILU if c["act"] == "silu" else binding.ACT_GELU)


def work(case):
    """Every input once, every result once; the products of Algorithm 1 with the saved matrix, of the gradient from the
    factors and of the rebuilt matrix (the orthonormalisation is left out: it depends on the method)."""
    n, d, r, g, t = case["n"], case["d"], case["r"], case["g"], case["t"]
    es = 2 if case["dtype"] == "bf16" else 4
    x, uv = n * d * es, (n + d) * r * es
    if case["kind"] in ("step", "prenorm"):
        nbytes = x + uv + 4 * r + n * g * es + 4 * d * g
        flops = 4.0 * n * d * r * (1 + t) + 2.0 * (n + d) * r * g
        if case["norm"]:
            nbytes += x + 4 * n + 2 * d * es + (4 * n if case["norm"] == "layer" else 0)
        if case["norm"] == "rms":
            nbytes += 2 * x
            flops += 4.0 * n * d * r
        return {"bytes": nbytes, "flops": flops}
    if case["kind"] == "wgrad":
        return {"bytes": uv + n * g * es + 4 * d * g, "flops": 2.0 * (n + d) * r * g}
    return {"bytes": uv + x * (2 if case["kind"] == "act" else 1), "flops": 2.0 * n * d * r}


def tolerance(case):
    """Four times what was seen against the same pass in 64 bits (an exact QR with a positive diagonal, so that the
    factors themselves compare entry by entry).  bf16 compression: the factors and the gradients are off by 1.7e-3 to
    3.0e-3 of their norm, the rounding of two bf16 factors, single entries by up to 2.1e-2; a rebuilt matrix and a
    gradient through it, from given factors, by 1.7e-3, one rounding.  fp32: V, dW and U V by 1e-7 to 1e-6; U by up to
    1.4e-4, because the last directions of the sketch are small.  dW from given factors: at most 1.5e-6 in either type."""
    if case["kind"] == "wgrad":
        return {"rel": 1e-5, "max": 5e-5}
    if case["dtype"] == "f32":
        return {"rel": 6e-4, "max": 8e-3} if case["kind"] == "step" else {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.1} if case["kind"] in ("step", "prenorm") else {"rel": 7e-3, "max": 0.03}
