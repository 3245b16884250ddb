"""Cases of use of the library: what one GPU of an AB-Training job has it do, over the sizes it has it done at.

A training cycle spends its steps in the factorised layer (forward, backward), its synchronisations in
mean -> split -> recombination, its full-rank phases in the dense layer and in the decomposition of the dense
weights, and every step in the optimizer.  Each listed case is one of those calls at a size of this repository's
workloads (ViT-B/16, ResNet-50 layer3, VGG16, the small fp32 layer) or at the edge of the range: one image, a
batch that fills the GPU, rows and widths that are multiples of no tile.  `draw` gives more of the same ranges.

Singular vectors are determined up to sign, and within a group of close values up to rotation, so the factors a
split returns are not comparable element by element.  A pass over a split therefore ends where the method goes
on: with the recombination W = A B of the factors (Algorithm 1), which is what they determine, beside the
singular values and the kept rank.
"""
import math

import torch

from paper_2405_01067_b200 import binding as ab

BF16, F32 = "bf16", "f32"

# 12 blocks of four attention matrices and the MLP pair
VIT_BLOCK = ((768, 768, 4), (3072, 768, 1), (768, 3072, 1))


def listed():
    return [
        # The small fp32 layer: seven launches of microseconds each; what a step costs when nothing is large.
        {"name": "layer_fp32_64_rows", "op": "layer", "m": 256, "n": 512, "r": 32, "rows": 64, "dtype": F32, "pass": "train"},
        # Inference on one image: 197 tokens through one factorised MLP layer, two row blocks on 148 SMs.
        {"name": "layer_infer_one_image", "op": "layer", "m": 3072, "n": 768, "r": 192, "rows": 197, "dtype": BF16,
         "pass": "forward"},
        # The headline step: forward and backward of both MLP layers of ViT-B/16 on a batch of 256 images.
        {"name": "vit_mlp_pair_train", "op": "mlp", "m": 3072, "n": 768, "r": 192, "rows": 50432, "dtype": BF16, "pass": "train"},
        # A group that trains only B (dX and dB wanted), last batch of an epoch, classifier-like widths: odd row
        # count, widths and rank that are multiples of 8 and of no tile.
        {"name": "layer_ragged_b_group", "op": "layer", "m": 1000, "n": 776, "r": 120, "rows": 6173, "dtype": BF16,
         "pass": "b_group"},
        # ResNet-50 layer3 3x3 convolution on NHWC activations, batch 128.
        {"name": "conv_resnet_train", "op": "conv", "batch": 128, "hw": 14, "c": 256, "m": 256, "r": 128},
        # VGG16 on CIFAR-10, 4x4 images, batch 1024, at a high compression: skinny products.
        {"name": "conv_vgg_train", "op": "conv", "batch": 1024, "hw": 4, "c": 512, "m": 512, "r": 32},
        # A full-rank step (warm-up, rebound) of the ViT MLP layer.
        {"name": "dense_vit_train", "op": "dense", "m": 3072, "n": 768, "rows": 50432},
        # The optimizer on all factors of ViT-B/16 in one arena, with the bf16 copy the layers read.
        {"name": "adamw_vit_factors", "op": "adamw", "count": 31850496},
        # Group synchronisation of all of ViT-B/16: 72 matrices, 8 copies, rank rule at 0.1.
        {"name": "sync_vit_model", "op": "sync", "blocks": 12, "m": 0, "n": 0, "r": 0, "copies": 8, "cutoff": 0.1, "dtype": F32},
        # Group synchronisation of one bf16 layer (VGG16 512x4608): a lone matrix, W wanted as well.
        {"name": "sync_vgg_layer", "op": "sync", "blocks": 0, "m": 512, "n": 4608, "r": 64, "copies": 4, "cutoff": 0.1,
         "dtype": BF16},
        # Decomposition of a dense trained weight: ViT MLP at rank 192 of 768.
        {"name": "split_vit_mlp", "op": "split", "m": 3072, "n": 768, "r": 192},
        # The same for a convolution weight whose short side is 256 (ResNet-50 layer3).
        {"name": "split_resnet_conv", "op": "split", "m": 256, "n": 2304, "r": 128},
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))
    return max(lo, min(hi, int(v) // step * step))


def draw(rng):
    op = rng.choice(["layer", "layer", "layer", "conv", "dense", "adamw", "sync", "split"])
    if op == "layer":
        if rng.random() < 0.2:      # fp32 layers are the small ones; any width, any rank
            m, n = _log_int(rng, 16, 1024), _log_int(rng, 16, 1024)
            return {"op": op, "m": m, "n": n, "r": _log_int(rng, 1, min(m, n, 256)), "rows": _log_int(rng, 1, 4096), "dtype": F32,
                    "pass": rng.choice(["train", "forward"])}
        m, n = _log_int(rng, 64, 3072, 8), _log_int(rng, 64, 3072, 8)
        return {"op": op, "m": m, "n": n, "r": _log_int(rng, 8, min(m, n, 256), 8), "rows": _log_int(rng, 1, 50432),
                "dtype": BF16, "pass": rng.choice(["train", "train", "b_group", "a_group", "forward"])}
    if op == "conv":
        hw = rng.choice([2, 4, 7, 8, 14, 28])
        c, m = _log_int(rng, 64, 512, 8), _log_int(rng, 64, 512, 8)
        return {"op": op, "batch": _log_int(rng, 1, max(1, 25088 // (hw * hw))), "hw": hw, "c": c, "m": m,
                "r": _log_int(rng, 8, min(m, 256), 8)}
    if op == "dense":
        return {"op": op, "m": _log_int(rng, 64, 3072, 8), "n": _log_int(rng, 64, 768, 8), "rows": _log_int(rng, 1, 50432)}
    if op == "adamw":
        return {"op": op, "count": _log_int(rng, 256, 31850496)}
    if op == "sync":
        m, n = _log_int(rng, 64, 3072, 8), _log_int(rng, 64, 3072, 8)
        dtype = rng.choice([F32, F32, BF16])
        return {"op": op, "blocks": rng.choice([0, 0, 1, 2]), "m": m, "n": n,
                "r": _log_int(rng, 8, min(m, n, 768) // 4, 8 if dtype == BF16 else 4),
                "copies": rng.randint(2, 8), "cutoff": rng.choice([0.05, 0.1, 0.2]), "dtype": dtype}
    short, long_ = _log_int(rng, 32, 768), _log_int(rng, 768, 3072)
    m, n = (short, long_) if rng.random() < 0.5 else (long_, short)
    return {"op": op, "m": m, "n": n, "r": _log_int(rng, 8, max(8, short // 2))}


# ------------------------------------------------------------------------------------------------ inputs

def _torch_dtype(name):
    return torch.bfloat16 if name == BF16 else torch.float32


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, shape, std=1.0, dtype=torch.float32):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(dtype)


def _orthonormal(g, rows, cols, count=1):
    return torch.linalg.qr(torch.randn((count, rows, cols), generator=g, device="cuda"))[0]


def _factors(g, m, n, r, sigma, count=1):
    """`count` factor pairs A = P diag(sigma)^(1/2), B = diag(sigma)^(1/2) Q^T, as a trained layer holds them."""
    h = sigma.sqrt()
    return (_orthonormal(g, m, r, count) * h).contiguous(), (h[:, None] * _orthonormal(g, n, r, count).transpose(1, 2)).contiguous()


def _layer_state(g, m, n, r, rows, dtype, what):
    """One factorised layer: activations and upstream gradient N(0, 1), a decaying spectrum on a flat floor."""
    td = _torch_dtype(dtype)
    dt = ab.AB_BF16 if dtype == BF16 else ab.AB_F32
    sigma = (0.9 ** torch.arange(r, device="cuda")).clamp(min=0.05) * (1.0 + 0.02 * (math.sqrt(m) + math.sqrt(n)))
    A, B = (t[0].to(td) for t in _factors(g, m, n, r, sigma))
    s = {"x": _normal(g, (rows, n), dtype=td), "A": A, "B": B, "y": torch.empty((rows, m), dtype=td, device="cuda"),
         "ws_f": ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_LAYER_FORWARD, rows, m, n, r, 1, dt), "cuda"), "pass": what}
    if what != "forward":
        s["dY"] = _normal(g, (rows, m), dtype=td)
        s["T"] = torch.empty((rows, r), dtype=td, device="cuda")
        s["want"] = {"train": ("dX", "dA", "dB"), "b_group": ("dX", "dB"), "a_group": ("dA",)}[what]
        s["dX"] = torch.empty((rows, n), dtype=td, device="cuda") if "dX" in s["want"] else None
        s["dA"] = torch.empty((m, r), device="cuda") if "dA" in s["want"] else None
        s["dB"] = torch.empty((r, n), device="cuda") if "dB" in s["want"] else None
        s["ws_b"] = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_LAYER_BACKWARD, rows, m, n, r, 1, dt), "cuda")
    return s


def _layer_run(s):
    if s["pass"] == "forward":
        ab.ab_layer_forward(s["x"], s["A"], s["B"], y=s["y"], ws=s["ws_f"])
        return {"y": s["y"]}
    ab.ab_layer_forward(s["x"], s["A"], s["B"], y=s["y"], T_save=s["T"], ws=s["ws_f"])
    ab.ab_layer_backward(s["x"], s["dY"], s["A"], s["B"], T_saved=s["T"], want=s["want"], dX=s["dX"], dA=s["dA"], dB=s["dB"],
                         ws=s["ws_b"])
    return {k: s[k] for k in ("y",) + s["want"]}


def _conv_state(g, c):
    """Post-ReLU-like activations (half normal), Kaiming-sized weight spectrum."""
    b, hw, ch, m, r = c["batch"], c["hw"], c["c"], c["m"], c["r"]
    n = 9 * ch
    sigma = math.sqrt(2.0 / n) * (math.sqrt(n) + math.sqrt(m) * torch.linspace(1.0, 0.0, r, device="cuda"))
    A, B = (t[0].to(torch.bfloat16) for t in _factors(g, m, n, r, sigma))
    return {"x": _normal(g, (b, hw, hw, ch)).abs().to(torch.bfloat16), "dY": _normal(g, (b, hw, hw, m), dtype=torch.bfloat16),
            "A": A, "B": B, "y": torch.empty((b, hw, hw, m), dtype=torch.bfloat16, device="cuda"),
            "T": torch.empty((b * hw * hw, r), dtype=torch.bfloat16, device="cuda"),
            "dX": torch.empty((b, hw, hw, ch), dtype=torch.bfloat16, device="cuda"), "dA": torch.empty((m, r), device="cuda"),
            "dB": torch.empty((r, n), device="cuda"), "ws": ab.workspace(ab.ab_conv3x3_workspace_bytes(b, hw, hw, ch, m, r), "cuda")}


def _conv_run(s):
    ab.ab_conv3x3_forward(s["x"], s["A"], s["B"], y=s["y"], T_save=s["T"], ws=s["ws"])
    ab.ab_conv3x3_backward(s["x"], s["dY"], s["A"], s["B"], T_saved=s["T"], dX=s["dX"], dA=s["dA"], dB=s["dB"], ws=s["ws"])
    return {k: s[k] for k in ("y", "dX", "dA", "dB")}


def _dense_state(g, c):
    m, n, rows, td = c["m"], c["n"], c["rows"], torch.bfloat16
    return {"x": _normal(g, (rows, n), dtype=td), "dY": _normal(g, (rows, m), dtype=td), "W": _normal(g, (m, n), 0.02, td),
            "y": torch.empty((rows, m), dtype=td, device="cuda"), "dX": torch.empty((rows, n), dtype=td, device="cuda"),
            "dW": torch.empty((m, n), device="cuda"),
            "ws_f": ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_DENSE_FORWARD, rows, m, n, 0, 1, ab.AB_BF16), "cuda"),
            "ws_b": ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_DENSE_BACKWARD, rows, m, n, 0, 1, ab.AB_BF16), "cuda")}


def _dense_run(s):
    ab.ab_dense_forward(s["x"], s["W"], y=s["y"], ws=s["ws_f"])
    ab.ab_dense_backward(s["x"], s["dY"], s["W"], dX=s["dX"], dW=s["dW"], ws=s["ws_b"])
    return {k: s[k] for k in ("y", "dX", "dW")}


def _adamw_state(g, c):
    n = c["count"]
    m = _normal(g, (n,), 1e-2)
    return {"p": _normal(g, (n,), 0.05), "g": _normal(g, (n,), 1e-2), "m": m, "v": m * m + 1e-6,
            "p_bf16": torch.empty((n,), dtype=torch.bfloat16, device="cuda")}


def _adamw_run(s):
    ab.ab_adamw_step(s["p"], s["g"], s["m"], s["v"], lr=1e-4, step=100, param_bf16=s["p_bf16"])
    return {k: s[k] for k in ("p", "m", "v", "p_bf16")}


def _sync_shapes(c):
    """(m, n, r, how many) of the model's matrices: whole ViT blocks and / or one layer of its own."""
    shapes = [(m, n, min(m, n) // 4, k * c["blocks"]) for m, n, k in VIT_BLOCK] if c["blocks"] else []
    return shapes + ([(c["m"], c["n"], c["r"], 1)] if c["m"] else [])


def _sync_state(g, c):
    """K copies of every factor pair: the planted pair (spectrum exp(-i/64)) and N(0, var 1e-3) of each group.
    Kept ranks, singular values and recombined weights lie in packed arrays, one per kind and shape."""
    td, K = _torch_dtype(c["dtype"]), c["copies"]
    std = math.sqrt(1e-3)
    Ac, Bc, W, Wr = [], [], [], []
    for m, n, r, count in _sync_shapes(c):
        A, B = _factors(g, m, n, r, torch.exp(-torch.arange(r, device="cuda") / 64.0), count)
        Wr.append(torch.empty((count, m, n), device="cuda"))
        for i in range(count):
            Ac.append((A[i] + _normal(g, (K, m, r), std)).to(td))
            Bc.append((B[i] + _normal(g, (K, r, n), std)).to(td))
            W.append(Wr[-1][i])
    plan = ab.SyncPlan(Ac, Bc, c["cutoff"], want_W=not c["blocks"])
    sigma = torch.empty((sum(t.numel() for t in plan.sigma),), device="cuda")
    at = 0
    for i, t in enumerate(plan.sigma):
        plan.sigma[i] = sigma[at:at + t.numel()]
        plan.descs[i].sigma = plan.sigma[i].data_ptr()
        at += t.numel()
    dt = ab.AB_BF16 if c["dtype"] == BF16 else ab.AB_F32
    need = max(ab.ab_workspace_bytes(ab.AB_OP_RECOMBINE, 0, m, n, r, 1, dt) for m, n, r, _ in _sync_shapes(c))
    return {"plan": plan, "W": W, "Wr": Wr, "sigma": sigma, "ws": ab.workspace(need, "cuda")}


def _sync_run(s):
    plan = s["plan"]
    ab.ab_group_sync(plan)
    for A, B, W in zip(plan.A_out, plan.B_out, s["W"]):
        ab.ab_recombine(A, B, W=W, ws=s["ws"])
    return {"sigma": s["sigma"], "rank": plan.r_out, "status": plan.status, "W": s["Wr"], "W_mean": plan.W_out}


def _split_state(g, c):
    """A dense weight: N(0, 0.02^2) plus a planted decaying spectrum 0.9^i."""
    m, n, r = c["m"], c["n"], c["r"]
    s = min(m, n)
    sigma = 0.9 ** torch.arange(s, device="cuda")
    W = 0.02 * torch.randn((m, n), generator=g, device="cuda") + (_orthonormal(g, m, s)[0] * sigma) @ _orthonormal(g, n, s)[0].T
    return {"W": W.contiguous(), "r": r, "Wr": torch.empty((m, n), device="cuda"),
            "ws": ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_SVD_SPLIT, 0, m, n, r, 1, ab.AB_F32), "cuda"),
            "ws_r": ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_RECOMBINE, 0, m, n, r, 1, ab.AB_F32), "cuda")}


def _split_run(s):
    A, B, sigma, rank, status = ab.ab_svd_split(s["W"], s["r"], 0.02, ws=s["ws"])
    ab.ab_recombine(A, B, W=s["Wr"], ws=s["ws_r"])
    return {"sigma": sigma, "rank": rank, "status": status, "W": s["Wr"]}


def prepare(case, seed):
    g, op = _gen(seed), case["op"]
    if op == "mlp":      # W1 is m x n, W2 is n x m: each on activations of its own
        a = (case["r"], case["rows"], case["dtype"], case["pass"])
        s = {"layers": [_layer_state(g, case["m"], case["n"], *a), _layer_state(g, case["n"], case["m"], *a)]}
    elif op == "layer":
        s = _layer_state(g, case["m"], case["n"], case["r"], case["rows"], case["dtype"], case["pass"])
    else:
        s = {"conv": _conv_state, "dense": _dense_state, "adamw": _adamw_state, "sync": _sync_state, "split": _split_state}[op](g, case)
    s["op"] = op
    return s


def run(state):
    if state["op"] == "mlp":
        return [_layer_run(s) for s in state["layers"]]
    return {"layer": _layer_run, "conv": _conv_run, "dense": _dense_run, "adamw": _adamw_run, "sync": _sync_run,
            "split": _split_run}[state["op"]](state)


# ------------------------------------------------------------------------------------------------ yardsticks

def _layer_work(m, n, r, rows, dtype, what):
    e = 2 if dtype == BF16 else 4
    mn, pair = m + n, rows * r * 2
    if what == "forward":
        return {"bytes": e * (rows * mn + r * mn), "flops": pair * mn}
    reads = rows * (n + m) + r * mn                                    # x, dY, A, B
    writes = rows * m + (rows * n if what != "a_group" else 0)          # y, dX
    grads = {"train": r * mn, "b_group": r * n, "a_group": r * m}[what]   # dA, dB in fp32
    flops = {"train": 3 * mn, "b_group": 2 * mn + n, "a_group": mn + m}[what]
    return {"bytes": e * (reads + writes) + 4 * grads, "flops": pair * flops}


def work(case):
    op = case["op"]
    if op in ("layer", "mlp"):
        w = _layer_work(case["m"], case["n"], case["r"], case["rows"], case["dtype"], case["pass"])
        if op == "mlp":
            w2 = _layer_work(case["n"], case["m"], case["r"], case["rows"], case["dtype"], case["pass"])
            w = {k: w[k] + w2[k] for k in w}
        return w
    if op == "conv":
        px, c, m, r = case["batch"] * case["hw"] ** 2, case["c"], case["m"], case["r"]
        return {"bytes": 2 * (2 * px * (c + m) + r * (m + 9 * c)) + 4 * r * (m + 9 * c), "flops": 6 * px * r * (m + 9 * c)}
    if op == "dense":
        m, n, rows = case["m"], case["n"], case["rows"]
        return {"bytes": 2 * (2 * rows * (m + n) + m * n) + 4 * m * n, "flops": 6 * rows * m * n}
    if op == "adamw":
        return {"bytes": 30 * case["count"], "flops": 12 * case["count"]}
    if op == "sync":
        e, b, f = (2 if case["dtype"] == BF16 else 4), 0, 0
        for m, n, r, count in _sync_shapes(case):
            # copies in, factors and recombined W out; mean, two Gram matrices, the split of an r x r core, the new factors, W
            b += count * (e * (case["copies"] + 1) * r * (m + n) + 4 * m * n * (1 if case["blocks"] else 2))
            f += count * (case["copies"] * r * (m + n) + 4 * r * r * (m + n) + 9 * r ** 3 + 2 * m * n * r * (1 if case["blocks"] else 2))
        return {"bytes": b, "flops": f}
    m, n, r = case["m"], case["n"], case["r"]
    s, l = min(m, n), max(m, n)
    # Gram matrix, its tridiagonal form, the leading vectors, the long factor, W = A B
    return {"bytes": 4 * (2 * m * n + r * (m + n)), "flops": 2 * l * s * s + 4 * s ** 3 // 3 + 2 * r * s * s + 4 * m * n * r}


def tolerance(case):
    """About four times what the results are off from float64 (relative 2-norm)."""
    op = case["op"]
    if op in ("layer", "mlp"):      # bf16: 2.3e-3 (T rounded, result rounded); fp32: sums of up to 4096 products
        return {"rel": 1e-2} if case["dtype"] == BF16 else {"rel": 5e-6}
    if op == "conv":                # as the bf16 layer
        return {"rel": 1e-2}
    if op == "dense":               # 1.7e-3: the rounding of a bf16 result
        return {"rel": 7e-3}
    if op == "adamw":               # max: one rounding of the bf16 copy
        return {"rel": 1e-6, "max": 1e-2}
    if op == "sync":                # bf16: 2.4e-3 (factors rounded); fp32: 3e-5
        return {"rel": 1e-2} if case["dtype"] == BF16 else {"rel": 1.2e-4}
    # The values themselves are good to 1e-7.  The product is as well determined as the gap behind the last kept
    # value: the bulk of this spectrum is dense, and 2e-5 to 8e-4 was seen over the sizes.
    return {"rel": 3e-3}
