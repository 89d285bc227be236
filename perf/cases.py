"""The workloads the library is timed on: what a user of BigBird attention has it do, through its public entry points.

Shapes are those of this repository's own workloads (``synth.py``), tests and benchmark: 12 x 64 heads (base) and
16 x 64 (large), 4096 tokens, 64-token blocks with 3 window, 2 global and 3 random blocks; the ETC variants; the
long 16384-token sequence; the fp32 path with its other block sizes and head dimensions.  Queries, keys, values and
output gradients are i.i.d. Gaussians, standing in for projected activations: scores scaled by 1/sqrt(D) are then
distributed like N(0, sigma^4).

A case is a dict of plain values:
    kind     "fwd": bigbird_attn_fwd;  "static": bigbird_attn_fwd_static (serving without allocations);
             "train": bigbird_attn_fwd, then bigbird_attn_bwd on its results (one layer's part of a training step)
    dtype    "bf16" or "fp32";  B, H, nb (key blocks; N = nb * b), D, b, w, g, r, mode (0 = ITC, 1 = ETC)
    sigma    standard deviation of the entries of q, k and v
    lo, hi   valid tokens of the shortest and of the longest sequence of the batch (the others lie evenly between,
             in an order drawn from the seed); hi = 0: no key-padding mask
    gtok     > 0: only this many of the g * b leading global slots hold a token, the rest is masked
"""
import math

import numpy as np
import torch

import paper_2007_14062_b200 as bb

LAYOUT_SEED = 1


def _case(kind, dtype, B, H, nb, D=64, b=64, w=3, g=2, r=3, mode=0, sigma=1.0, lo=0, hi=0, gtok=0):
    return dict(kind=kind, dtype=dtype, B=B, H=H, nb=nb, D=D, b=b, w=w, g=g, r=r, mode=mode, sigma=sigma, lo=lo, hi=hi,
                gtok=gtok)


def listed():
    named = [
        # the smallest call: a short fp32 sequence, as in a unit test or a debugging session of a model; latency only
        ("fp32_tiny_fwd", _case("fwd", "fp32", 1, 2, 8)),
        # serving: one request of 3001 tokens padded to the model's 4096, on the entry point that allocates nothing
        ("serve_one_static", _case("static", "bf16", 1, 12, 64, lo=3001, hi=3001)),
        # inference or evaluation with the base model: eight full sequences
        ("base_fwd", _case("fwd", "bf16", 8, 12, 64)),
        # the ETC variant: 128 extra global tokens in front of 4096, no random blocks
        ("etc_fwd", _case("fwd", "bf16", 8, 12, 66, r=0, mode=1)),
        # one long document of 13000 tokens in a 16384-token model
        ("long_fwd", _case("fwd", "bf16", 1, 12, 256, sigma=0.5, lo=13000, hi=13000)),
        # the large model on a ragged batch: the largest forward call
        ("large_ragged_fwd", _case("fwd", "bf16", 16, 16, 64, lo=1024, hi=4096)),
        # fine-tuning on short texts: a small training micro-batch with padding
        ("short_train", _case("train", "bf16", 2, 12, 16, lo=333, hi=1024)),
        # pretraining with the base model: full sequences, forward and backward
        ("base_train", _case("train", "bf16", 8, 12, 64)),
        # fine-tuning the large model on documents of different lengths, none a multiple of the block size
        ("large_ragged_train", _case("train", "bf16", 3, 16, 64, lo=1001, hi=3999)),
        # training on one long document
        ("long_train", _case("train", "bf16", 1, 12, 256, sigma=0.5, lo=13000, hi=13000)),
        # the paper's ETC base setting, in fp32: block 84, 230 global tokens in three blocks, no random blocks
        ("etc84_fp32_train", _case("train", "fp32", 2, 12, 52, b=84, g=3, r=0, mode=1, lo=4368, hi=4368, gtok=230)),
        # fp32 evaluation with 128-wide heads on a small ragged batch
        ("fp32_d128_fwd", _case("fwd", "fp32", 2, 8, 40, D=128, lo=1500, hi=2560)),
    ]
    return [dict(case, name=name) for name, case in named]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# The most a drawn case of each kind may cost: B * H * nb * b * D, as in the largest listed case of that kind.
_MOST = {("fwd", "bf16"): 16 * 16 * 4096 * 64, ("static", "bf16"): 8 * 12 * 4096 * 64, ("train", "bf16"): 8 * 12 * 4096 * 64,
         ("fwd", "fp32"): 2 * 12 * 4368 * 64, ("train", "fp32"): 2 * 12 * 4368 * 64}


def draw(rng):
    """One more case of the same ranges."""
    kind, dtype = rng.choice([("fwd", "bf16"), ("fwd", "bf16"), ("static", "bf16"), ("train", "bf16"), ("train", "bf16"),
                              ("train", "fp32"), ("fwd", "fp32")])
    while True:
        D, b = 64, 64                   # what the bf16 forward pass takes
        if dtype == "fp32":
            D, b = rng.choice([32, 64, 64, 128]), rng.choice([16, 64, 64, 84, 169])
        most_nb = {"fwd": 256, "static": 96, "train": 256}[kind]
        nb = _log_int(rng, 6, max(8, most_nb * 64 // b if b >= 64 else 128))
        B = _log_int(rng, 1, 16 if kind == "fwd" else 8)
        H = rng.choice([2, 5, 8, 12, 12, 16, 16])
        if B * H * nb * b * D <= _MOST[(kind, dtype)]:
            break
    mode = rng.choice([0, 0, 1])
    g = rng.choice([1, 2, 2, 3])
    case = _case(kind, dtype, B, H, nb, D=D, b=b, w=rng.choice([3, 3, 3, 5]), g=g, r=rng.choice([0, 2, 3, 3]), mode=mode,
                 sigma=rng.choice([0.5, 1.0, 1.0, 1.5]))
    N = nb * b
    if rng.random() < 0.6:
        hi = rng.choice([N, rng.randint(max(b, N // 2), N)])
        lo = rng.randint(max(1, hi // 4), hi)
        if nb > 96:                     # batches of long documents are made of ones of about the same length
            hi = rng.randint((nb - 1) // 32 * 32 * b + 1, N)
            lo = rng.randint((nb - 1) // 32 * 32 * b + 1, hi)
        case.update(lo=lo, hi=hi)
    return case


def _lengths(case):
    B = case["B"]
    return np.round(np.linspace(case["lo"], case["hi"], B) if B > 1 else np.array([case["hi"]])).astype(np.int64)


def _mask(case, lengths):
    """uint8 [B, N], 1 = token, or None if the case has no padding."""
    if not case["hi"]:
        return None
    N = case["nb"] * case["b"]
    mask = (np.arange(N)[None, :] < lengths[:, None]).astype(np.uint8)
    if case["gtok"]:
        mask[:, case["gtok"]:case["g"] * case["b"]] = 0
    return mask


def _layout(case):
    return bb.bigbird_build_layout(case["nb"] * case["b"], case["b"], case["w"], case["g"], case["r"], LAYOUT_SEED, case["H"],
                                   case["mode"])


def prepare(case, seed):
    B, H, N, D = case["B"], case["H"], case["nb"] * case["b"], case["D"]
    dev, dtype = torch.device("cuda"), {"bf16": torch.bfloat16, "fp32": torch.float32}[case["dtype"]]
    gen = torch.Generator(device=dev).manual_seed(seed)

    def normal(sigma):
        return (torch.randn((B, H, N, D), generator=gen, device=dev) * sigma).to(dtype)

    mask = _mask(case, np.random.RandomState(seed % 2**32).permutation(_lengths(case)))
    s = {"kind": case["kind"], "layout": _layout(case), "scale": 1.0 / math.sqrt(D),
         "q": normal(case["sigma"]), "k": normal(case["sigma"]), "v": normal(case["sigma"]),
         "mask": None if mask is None else torch.from_numpy(mask).to(dev)}
    s["out"] = torch.empty_like(s["q"])
    s["lse"] = torch.empty((B, H, N), device=dev, dtype=torch.float32)
    if case["kind"] == "train":
        s["dout"] = normal(1.0)
        s["dq"], s["dk"], s["dv"] = (torch.empty_like(s["q"]) for _ in range(3))
    s["fwd"] = bb.bigbird_attn_fwd_static if case["kind"] == "static" else bb.bigbird_attn_fwd
    return s


def run(s):
    s["fwd"](s["q"], s["k"], s["v"], s["layout"], s["mask"], s["out"], s["lse"], s["scale"])
    if s["kind"] != "train":
        return {"out": s["out"], "lse": s["lse"]}
    bb.bigbird_attn_bwd(s["q"], s["k"], s["v"], s["out"], s["lse"], s["dout"], s["layout"], s["mask"], s["dq"], s["dk"], s["dv"],
                        s["scale"])
    return {k: s[k] for k in ("out", "lse", "dq", "dk", "dv")}


def work(case):
    """Bytes: every tensor of the call once (q, k, v, dout and the mask in; out, lse, dq, dk, dv out).  FLOPs: per attended
    (valid query, valid key) pair two products of D for the forward pass and five for the backward pass."""
    B, H, nb, b, D = (case[k] for k in ("B", "H", "nb", "b", "D"))
    mask = _mask(case, _lengths(case))
    valid = np.full((B, nb), b, dtype=np.int64) if mask is None else mask.reshape(B, nb, b).sum(axis=2, dtype=np.int64)
    layout = _layout(case)
    row_ptr, col_idx = layout.export()
    layout.close()
    rows = np.repeat(np.arange(H * nb), np.diff(row_ptr)) % nb
    pairs = int((valid[:, rows] * valid[:, col_idx]).sum())
    train = case["kind"] == "train"
    elements, size = B * H * nb * b * D, 2 if case["dtype"] == "bf16" else 4
    return {"bytes": (8 if train else 4) * elements * size + B * H * nb * b * 4 + (0 if mask is None else mask.size),
            "flops": pairs * D * (14 if train else 4)}


def tolerance(case):
    # about four times the largest error of any output against dense attention and its gradients in fp64 over such cases:
    # 2.4e-3 for bf16 (probabilities and results rounded to bf16), 1e-6 for fp32 (sums of up to some 6000 terms)
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 5e-6}
