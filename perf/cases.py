"""Performance cases: the sampling and encoding calls a user of this library makes, through the ctypes binding.

A program loads a model once and then decodes (latents -> samples, the Jacobi / sequential / selective policies) or
encodes (samples -> latents and log-determinant) batch after batch.  The model handle is therefore kept from one
`prepare` to the next while the architecture stays the same; latents, samples and labels come from the seed.
Architectures are those of `synth.CONFIGS` / `synth.MAF_CONFIGS` and, for odd sizes, variations of the class-conditional
one with another image grid and width.  Weights follow the recipe of `synth.make_weights` (same shapes, same standard
deviations), drawn with torch on the GPU because the full models have up to 0.8 billion of them.

Only samples, latents and log-determinants are compared: the sweep counts a call can also report are a by-product of
the stopping test and may differ by one where a sample's max|du| lands next to tau.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_24791_b200 import binding, synth

# Largest batch each architecture is loaded for (sizes its workspace and key/value cache).
MAX_BATCH = {"cfg1": 64, "cfg2": 256, "cfg3": 256, "cfg4": 16, "ragged": 64, "maf_ising": 100000, "maf_mnist": 1000}


def listed():
    return [
        # Smallest call: the tiny fp32 model, four samples; the cost is launches and the host loop.
        dict(name="tiny_fp32_selective_b4", model="cfg1", batch=4, call="inverse", policy="selective", tau=1e-5),
        # 32x32 sampling as configured: 256 tokens of width 512, batch 64, first block sequential, the others Jacobi.
        dict(name="small_selective_b64", model="cfg2", batch=64, call="inverse", policy="selective", tau=1e-3),
        # The same model behind a service that holds its data on the host, an odd batch, uniform Jacobi.
        dict(name="small_jacobi_host_b37", model="cfg2", batch=37, call="inverse_host", policy="jacobi", tau=1e-3),
        # Odd sizes: 9x9 patches = 81 tokens, width 256, ten classes, 13 samples.
        dict(name="ragged_selective_b13", model="ragged", batch=13, call="inverse", policy="selective", tau=1e-3, rows=9, cols=9,
             width=256),
        # One image at a time from the class-conditional model (64x64, 256 tokens, width 1024, 8 blocks x 8 layers):
        # the interactive end of its batch range, where weights stream past few rows.
        dict(name="classcond_jacobi_b1", model="cfg3", batch=1, call="inverse", policy="jacobi", tau=1e-3),
        # Token-by-token decoding with the key/value cache, the baseline the paper compares with, at a small batch.
        dict(name="classcond_sequential_b8", model="cfg3", batch=8, call="inverse", policy="sequential", tau=0.0),
        # The headline workload: class-conditional sampling, batch 64, selective policy.
        dict(name="classcond_selective_b64", model="cfg3", batch=64, call="inverse", policy="selective", tau=1e-3),
        # Bulk generation at the loose threshold of the policy table: the largest batch, uniform Jacobi.
        dict(name="classcond_jacobi_b256", model="cfg3", batch=256, call="inverse", policy="jacobi", tau=1e-2),
        # Encoding: data to latents and log-determinant (one causal pass per block), batch 64.
        dict(name="classcond_forward_b64", model="cfg3", batch=64, call="forward", policy="", tau=0.0),
        # 256x256 sampling as configured: 1024 tokens, batch 16 (attention and the key/value cache weigh most here).
        dict(name="long_selective_b16", model="cfg4", batch=16, call="inverse", policy="selective", tau=1e-3),
        # MLP-based flow on a 16x16 lattice, 100 000 samples per call (the Boltzmann-generator use).
        dict(name="maf_ising_jacobi_b100000", model="maf_ising", batch=100000, call="inverse", policy="jacobi", tau=1e-3),
        # MLP-based flow on 28x28 images, 100 samples.
        dict(name="maf_mnist_jacobi_b100", model="maf_mnist", batch=100, call="inverse", policy="jacobi", tau=1e-3),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more call of the same ranges: any of the models, policies, thresholds and directions, batches spread over the
    logarithm of the model's range (upper ends chosen so that no call costs more than the largest listed one)."""
    model = rng.choice(["cfg1", "cfg2", "cfg3", "cfg4", "ragged", "maf_ising", "maf_mnist"])
    tau = rng.choice([1e-4, 1e-5]) if model == "cfg1" else rng.choice([1e-2, 1e-3, 1e-4])
    call = rng.choice(["inverse", "inverse", "inverse", "forward"])
    if model in synth.MAF_CONFIGS:
        policy = rng.choice(["jacobi", "jacobi", "sequential"])
        lo, hi = (100, 100000) if model == "maf_ising" else (10, 1000)
        if call == "inverse" and policy == "sequential":
            hi = min(hi, 4096)
        case = dict(model=model, batch=_log_int(rng, lo, hi), call=call, policy=policy, tau=tau)
    else:
        policy = rng.choice(["selective", "jacobi", "sequential"] if model != "cfg4" else ["selective", "jacobi"])
        if call == "inverse" and model != "cfg1" and rng.random() < 0.25:
            call = "inverse_host"
        hi = MAX_BATCH[model]
        if model == "cfg3" and call != "forward":
            hi = 64 if policy == "sequential" else 96 if policy == "selective" or tau < 1e-2 else 256
        case = dict(model=model, batch=_log_int(rng, 1, hi), call=call, policy=policy, tau=tau)
        if model == "ragged":
            case.update(rows=rng.randint(5, 20), cols=rng.randint(5, 20), width=rng.choice([128, 256, 512]))
    if case["call"] == "forward":
        case.update(policy="", tau=0.0)
    elif case["policy"] == "sequential":
        case["tau"] = 0.0
    return case


def _config(case):
    if case["model"] in synth.MAF_CONFIGS:
        return synth.maf_config(case["model"])
    if case["model"] == "ragged":
        return synth.config("cfg3", H=4 * case["rows"], W=4 * case["cols"], n_blocks=2, n_layers=2, width=case["width"],
                            n_heads=case["width"] // 64, n_classes=10)
    return synth.config(case["model"])


# ---- weights -------------------------------------------------------------------------------------------------------
def _fill(name, shape, out, gen, cfg, maf):
    """One tensor of a block in `out` (flat, on the GPU), with the standard deviations of synth's seeded weights."""
    base = name.split(".")[-1]
    out.normal_(generator=gen)
    if maf:
        std = {"w1": 2.0 / math.sqrt(shape[-1]), "w2": 2.0 / math.sqrt(shape[-1]), "w3": 0.1 / math.sqrt(shape[-1] / 2.0)}
        out.mul_(std.get(name, 0.02))
        matrix = name.startswith("w")
    else:
        matrix = base.startswith("w_")
        if base == "w_out":
            out.mul_(0.1 / math.sqrt(cfg["width"]))
        elif matrix:
            out.mul_(math.sqrt(2.0 / (shape[0] + shape[1])))
        else:
            out.mul_(0.02)
            if base in ("ln1_g", "ln2_g", "lnf_g"):
                out.add_(1.0)
    if matrix and cfg["dtype"] == 1:
        out.copy_(out.bfloat16())


def _weight_blob(cfg, maf):
    specs = synth.maf_tensor_specs(cfg) if maf else synth.block_tensor_specs(cfg)
    header = (synth.pack_maf_blob if maf else synth.pack_blob)(cfg, [])   # no blocks: the header alone
    per_block = sum(int(np.prod(shape)) for _, shape in specs)
    blob = np.empty(header.nbytes + 4 * per_block * cfg["n_blocks"], dtype=np.uint8)
    blob[: header.nbytes] = header
    floats = torch.from_numpy(blob[header.nbytes:].view(np.float32)).view(cfg["n_blocks"], per_block)
    gen = torch.Generator(device="cuda").manual_seed(synth.WEIGHT_SEED)
    flat = torch.empty(per_block, device="cuda")
    for g in range(cfg["n_blocks"]):
        at = 0
        for name, shape in specs:
            n = int(np.prod(shape))
            _fill(name, shape, flat[at:at + n], gen, cfg, maf)
            at += n
        floats[g].copy_(flat)
    return blob


class _Model:
    """A loaded model; released when neither a state nor the cache below refers to it any more."""

    def __init__(self, cfg, maf, max_batch):
        self.handle = (binding.tf_maf_load if maf else binding.tf_load)(cfg, _weight_blob(cfg, maf), max_batch)

    def __del__(self):
        if getattr(self, "handle", None) is not None:
            binding.tf_free(self.handle)


_loaded = {}   # at most one entry: the model of the last case, kept as a sampling program keeps its own


def _model(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k in ("model", "rows", "cols", "width")))
    if key not in _loaded:
        _loaded.clear()
        _loaded[key] = _Model(_config(case), case["model"] in synth.MAF_CONFIGS, MAX_BATCH[case["model"]])
    return _loaded[key]


# ---- one call ------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    cfg, B = _config(case), case["batch"]
    maf = case["model"] in synth.MAF_CONFIGS
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    shape = (B, cfg["D"]) if maf else (B, cfg["C"], cfg["H"], cfg["W"])
    # latents are N(0, 1) * z_scale; with these weights samples keep about that scale, so `forward` takes the same
    source = torch.randn(shape, generator=gen, device="cuda") * cfg["z_scale"]
    state = dict(case=case, model=_model(case), batch=B, maf=maf, source=source, result=torch.empty_like(source), labels=None)
    if not maf:
        K = cfg["n_blocks"]
        state["policy"] = {"selective": [0] + [1] * (K - 1), "jacobi": [1] * K, "sequential": [0] * K, "": None}[case["policy"]]
        if cfg["n_classes"]:
            state["labels"] = torch.randint(0, cfg["n_classes"], (B,), generator=gen, device="cuda", dtype=torch.int32)
    state["max_iters"] = (cfg["D"] if maf else synth.seq_len(cfg)) + 1
    if case["call"] == "forward":
        state["logdet"] = torch.empty(B, device="cuda")
    if case["call"] == "inverse_host":
        for k in ("source", "result", "labels"):
            state[k] = None if state[k] is None else state[k].cpu().pin_memory()
    return state


def run(s):
    c, m, B = s["case"], s["model"].handle, s["batch"]
    if c["call"] == "forward":
        if s["maf"]:
            binding.tf_maf_forward(m, s["source"], B, s["result"], s["logdet"])
        else:
            binding.tf_forward(m, s["source"], s["labels"], B, s["result"], s["logdet"])
        return s["result"], s["logdet"]
    if s["maf"]:
        if c["policy"] == "sequential":
            binding.tf_maf_inverse_sequential(m, s["source"], B, s["result"])
        else:
            binding.tf_maf_inverse_jacobi(m, s["source"], B, c["tau"], s["max_iters"], 0, s["result"])
    elif c["call"] == "inverse_host":
        binding.tf_inverse_jacobi_host(m, s["source"], s["labels"], B, s["policy"], c["tau"], s["max_iters"], 0, s["result"])
    elif c["policy"] == "sequential":
        binding.tf_inverse_sequential(m, s["source"], s["labels"], B, s["result"])
    else:
        binding.tf_inverse_jacobi(m, s["source"], s["labels"], B, s["policy"], c["tau"], s["max_iters"], 0, s["result"])
    return s["result"]


# ---- what a call cannot do without ---------------------------------------------------------------------------------
# Fewest sweeps with which nearly all samples of these seeded models pass the stopping test (the largest count of a
# block is one or two higher).
SWEEPS = {1e-2: 5, 1e-3: 7, 1e-4: 8, 1e-5: 9}
MAF_SWEEPS = {1e-2: 3, 1e-3: 4, 1e-4: 5}


def work(case):
    """Every weight and every input read once, every output written once; FLOPs of the passes the policy asks for: one
    causal pass per block when encoding or decoding sequentially, SWEEPS passes per Jacobi block."""
    cfg, B, K = _config(case), case["batch"], _config(case)["n_blocks"]
    esz = 2 if cfg["dtype"] == 1 else 4
    if case["model"] in synth.MAF_CONFIGS:
        D, H = cfg["D"], cfg["hidden"]
        weights = K * (D * H + H * H + 2 * D * H)
        values = B * D
        # sequential decoding without a cache: dimension i needs its own pass, D of them per layer
        passes = K * (1 if case["call"] == "forward" else D if case["policy"] == "sequential" else MAF_SWEEPS[case["tau"]])
        flops = passes * B * 2.0 * (D * H + H * H + 2 * D * H)
    else:
        d, D, L, nl = cfg["width"], synth.token_dim(cfg), synth.seq_len(cfg), cfg["n_layers"]
        hid = cfg["mlp_ratio"] * d
        weights = K * (nl * (4 * d * d + 2 * d * hid) + 3 * D * d)
        values = B * L * D
        row = nl * (2.0 * (4 * d * d + 2 * d * hid) + 2.0 * d * L) + 6.0 * D * d
        n_seq = {"sequential": K, "selective": 1, "jacobi": 0, "": K}[case["policy"]]
        flops = B * L * row * (n_seq + (K - n_seq) * SWEEPS.get(case["tau"], 0))
    return {"bytes": float(esz * weights + 2 * 4 * values), "flops": float(flops)}


def tolerance(case):
    """fp32 engine: sums in fp32, and two runs may stop one sweep apart at tau <= 1e-4.  bf16 engine: operands in bf16
    (pairs of them once a sample is close to converged), sums and the state in fp32."""
    if _config(case)["dtype"] == 0:
        return {"rel": 2e-5, "max": 2e-4}
    return {"rel": 1e-2, "max": 1e-1}
