"""The work a user has this library do, as cases that can be timed and whose outputs can be compared.

Five kinds of case, one for each thing a pruning run of a model does with the library:

``hessian``  the calibration Hessian of a family of same-shape layers, from a forward pass's
             activations: token-major batches as the pass emits them (``layout = "tokens"``, one call
             a batch, ``beta = 1`` after the first) or one token-contiguous matrix (``"features"``);
``prune``    damped inverse, greedy loop and snapshots of such a family (``group = 1``: FFN neurons,
             otherwise attention heads of ``group`` columns);
``reshape``  a database of snapshots into the dense matrices a runtime executes;
``select``   one level per module under a run-time budget, for a batch of coefficient vectors;
``search``   the mutation search over those coefficients, one search per speedup target.

Sizes are those of ``workloads.CONFIGS`` (BERT-base, BERT-large, GPT-2 and the tiny layer), of the
tests, and the ragged ones that layers have once they have been pruned and are pruned again.
"""
from __future__ import annotations

import math

import torch

import paper_2302_04089_b200 as z

DAMP = 0.01
_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _hessian(name, layers, cols, tokens, batches=1, dtype="f32", layout="tokens"):
    return dict(name=name, kind="hessian", layers=layers, cols=cols, tokens=tokens, batches=batches,
                dtype=dtype, layout=layout)


def _prune(name, layers, rows, cols, group, levels):
    return dict(name=name, kind="prune", layers=layers, rows=rows, cols=cols, group=group, levels=levels)


def listed():
    return [
        # one small layer, one calibration batch: launches and host work count
        _hessian("hessian_tiny_f32", 1, 256, 2048),
        # BERT-base fc2, the calibration set arriving as eight fp32 batches of a forward pass
        _hessian("hessian_fc2_f32_batches", 12, 3072, 16384, batches=8),
        # GPT-2 mlp, bf16 activations of the whole calibration set in one call
        _hessian("hessian_mlp_bf16", 12, 3072, 131072, dtype="bf16", layout="features"),
        # one layer that an earlier pruning step left with 1322 neurons, fp16 activations
        _hessian("hessian_reshaped_f16", 1, 1322, 4099, dtype="f16"),
        # the tiny layer to three quarters removed: a chain of latencies
        _prune("prune_tiny", 1, 64, 256, 1, 4),
        # BERT-base fc2, all neurons, twelve levels: the benchmark's layers
        _prune("prune_fc2_base", 12, 768, 3072, 1, 12),
        # BERT-large fc2, all neurons, sixteen levels: the largest pruning run
        _prune("prune_fc2_large", 24, 1024, 4096, 1, 16),
        # layers reshaped to 1814 neurons by an earlier step of gradual pruning, the paper's level grid
        _prune("prune_fc2_reshaped", 12, 768, 1814, 1, 0),
        # BERT-base attention output projection, every head count
        _prune("prune_heads_base", 12, 768, 768, 64, 12),
        # the twelve-layer fc2 database into dense matrices, level by level
        dict(name="reshape_fc2", kind="reshape", layers=12, rows=768, cols=3072, group=1, levels=12),
        # a population of mutated coefficient vectors that a caller scores on its model
        dict(name="select_population", kind="select", candidates=1024, modules=24, buckets=10000),
        # the search over 1000 mutations for eight speedup targets
        dict(name="search_targets", kind="search", targets=8, modules=24, buckets=10000, steps=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hessian"] * 4 + ["neurons"] * 4 + ["heads"] * 2 + ["reshape", "select", "search"])
    if kind == "hessian":
        dtype, layout = rng.choice(sorted(_DTYPES)), rng.choice(["tokens", "tokens", "features"])
        layers, cols = _log(rng, 1, 24), _log(rng, 64, 4096)
        tokens = _log(rng, 256, min(131072, 1.2e12 / (layers * cols * cols), 4e9 / (layers * cols)))
        batches = rng.randint(1, 8) if layout == "tokens" and tokens >= 1024 else 1
        c = _hessian("", layers, cols, tokens, batches, dtype, layout)
    elif kind == "neurons":
        cols = _log(rng, 64, 4096)
        c = _prune("", _log(rng, 1, 24 if cols <= 2048 else 12), _log(rng, 32, 1024), cols, 1,
                   rng.choice([0, 4, 10, 12, 16]))
    elif kind == "heads":
        group, heads = rng.choice([32, 64, 64, 64, 80, 96, 128]), rng.randint(4, 16)
        heads = min(heads, 1280 // group)
        c = _prune("", _log(rng, 1, 24), _log(rng, 64, 1280), group * heads, group, 0)
    elif kind == "reshape":
        c = dict(kind="reshape", layers=_log(rng, 1, 24), rows=_log(rng, 32, 1024), cols=_log(rng, 64, 3072),
                 group=1, levels=rng.choice([4, 10, 12]))
    elif kind == "select":
        c = dict(kind="select", candidates=_log(rng, 1, 1024), modules=2 * rng.randint(6, 24),
                 buckets=_log(rng, 1000, 10000))
    else:
        c = dict(kind="search", targets=_log(rng, 1, 32), modules=2 * rng.randint(6, 12),
                 buckets=_log(rng, 1000, 10000), steps=_log(rng, 100, 1000))
    c.pop("name", None)
    return c


def _paper_sizes(G):
    """An FFN's sizes in the paper's database: relative steps of a tenth, and the dropped module."""
    return sorted({int(G * 0.9 ** i) for i in range(1, 43)} - {G} | {0}, reverse=True)


def _levels(case):
    """Strictly decreasing remaining-structure counts: ``levels`` evenly spaced ones, or the paper's grid."""
    G = case["cols"] // case["group"]
    if case["levels"] == 0:
        return _paper_sizes(G) if case["group"] == 1 else list(range(G - 1, -1, -1))
    if case["levels"] == 4:                  # the tiny layer stops at a quarter
        return sorted({G * i // 4 for i in (3, 2, 1)}, reverse=True)
    return sorted({G * i // case["levels"] for i in range(case["levels"])}, reverse=True)


def _activations(gen, recipe, cols, tokens):
    """[tokens, cols] fp32 on the GPU: inputs of an FFN's second layer (some neurons fire on nearly
    every token, some rarely: their biases differ), or of an attention output projection."""
    normal = lambda *s: torch.randn(*s, generator=gen, device="cuda")  # noqa: E731
    if recipe == "ffn":
        latent = max(16, cols // 4)
        pre = normal(tokens, latent) @ (normal(latent, cols) / latent ** 0.5)
        return torch.nn.functional.gelu(pre + (normal(cols) - 1.0))
    x = torch.nn.functional.layer_norm(normal(tokens, cols), (cols,))
    return x + normal(tokens, 64) @ normal(64, cols) / 8.0


def _database(case, seed):
    """Losses and run times of a model's modules, attention (every head count) and FFN (the paper's
    sizes) in turn, padded to the longer list."""
    gen = torch.Generator().manual_seed(seed)
    heads, sizes = list(range(12, -1, -1)), [3072] + _paper_sizes(3072)
    M, width = case["modules"], len(sizes)
    loss, time = torch.zeros(M, width), torch.zeros(M, width)
    count = torch.zeros(M, dtype=torch.int32)
    for m in range(M):
        opts, full, fixed = (heads, 4.0, 0.4) if m % 2 == 0 else (sizes, 11.9, 0.9)
        k = len(opts)
        kept = torch.tensor(opts, dtype=torch.float32) / opts[0]
        power = 1.5 + 2.0 * torch.rand(1, generator=gen)
        loss[m, :k] = (1.0 - kept) ** power * (1.0 + 0.01 * torch.rand(k, generator=gen))
        loss[m, k - 1] = 1.0
        time[m, :k] = torch.where(kept > 0, fixed + (full - fixed) * kept, torch.zeros(k))
        count[m] = k
    base = 0.5 + torch.rand(M, generator=gen)
    return dict(loss=(loss * base[:, None]).cuda(), base_loss=base.cuda(), time=time.cuda(),
                n_options=count.cuda()), float(time[:, 0].sum()), gen


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "hessian":
        gen = torch.Generator("cuda").manual_seed(seed)
        L, d, N, B = case["layers"], case["cols"], case["tokens"], case["batches"]
        dt = _DTYPES[case["dtype"]]
        if case["layout"] == "features":
            pitch = (N + 7) // 8 * 8          # rows start on 16-byte boundaries
            X = torch.zeros(L, d, pitch, dtype=dt, device="cuda")
            for l in range(L):
                X[l, :, :N] = _activations(gen, "ffn", d, N).t()
            st["X"] = X[:, :, :N]
        else:
            cuts = [N * b // B for b in range(B + 1)]
            st["A"] = [torch.stack([_activations(gen, "ffn", d, cuts[b + 1] - cuts[b]).to(dt) for _ in range(L)])
                       for b in range(B)]
    elif kind == "prune":
        gen = torch.Generator("cuda").manual_seed(seed)
        L, r, d = case["layers"], case["rows"], case["cols"]
        W = 0.02 * torch.randn(L, r, d, generator=gen, device="cuda")
        if case["group"] == 1:               # a trained layer's neurons do not all weigh the same
            W = W * torch.exp(0.5 * torch.randn(L, 1, d, generator=gen, device="cuda"))
        H = torch.empty(L, d, d, device="cuda")
        for l in range(L):
            A = _activations(gen, "ffn" if case["group"] == 1 else "attn", d, 4 * d + 8).double()
            S = A.t() @ A
            H[l] = (S + S.t()).float()        # 2 X X^T
        st["W"], st["H"], st["levels"] = W, H, _levels(case)
    elif kind == "reshape":
        gen = torch.Generator("cuda").manual_seed(seed)
        L, r, d, g = case["layers"], case["rows"], case["cols"], case["group"]
        st["levels"] = [v for v in _levels(case) if v > 0]
        order = torch.rand(L, d // g, generator=gen, device="cuda").argsort(dim=1)
        st["order"] = order.to(torch.int32)
        removed_at = order.argsort(dim=1).repeat_interleave(g, dim=1)
        W = 0.02 * torch.randn(L, 1, r, d, generator=gen, device="cuda")
        keep = torch.stack([removed_at >= d // g - v for v in st["levels"]], dim=1)
        st["W_snap"] = W * keep[:, :, None, :]
        st["previous"] = 0.02 * torch.randn(L, d, r, generator=gen, device="cuda")    # the layer that feeds it
    elif kind == "select":
        st["db"], total, gen = _database(case, seed)
        st["coef"] = (0.05 + 3.0 * torch.rand(case["candidates"], case["modules"], generator=gen)).cuda()
        st["budget"] = total / 2.0
    else:
        st["db"], total, gen = _database(case, seed)
        S, M, T = case["targets"], case["modules"], case["steps"]
        st["objective"] = (st["db"]["loss"] / st["db"]["base_loss"][:, None]
                           * (0.5 + torch.rand(M, 1, generator=gen)).cuda())
        st["coef0"] = torch.ones(S, M, device="cuda")
        st["budgets"] = torch.tensor([total / (1.5 + 0.5 * s) for s in range(S)], dtype=torch.float64).cuda()
        st["mask"] = (torch.rand(S, T, M, generator=gen) < 0.1).to(torch.uint8).cuda()
        st["values"] = (0.05 + 3.0 * torch.rand(S, T, M, generator=gen)).cuda()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "hessian":
        if case["layout"] == "features":
            return z.hessian_accumulate(st["X"])
        H = z.hessian_accumulate_tokens(st["A"][0])
        for A in st["A"][1:]:
            z.hessian_accumulate_tokens(A, H, beta=1.0)
        return H
    if kind == "prune":
        out = z.prune_layers(st["W"], st["H"], case["group"], DAMP, st["levels"])
        return {k: out[k] for k in ("W_snap", "loss", "base_loss", "order", "saliency", "layer_status")}
    if kind == "reshape":
        dense = []
        for slot, level in enumerate(st["levels"]):
            kept, status = z.kept_structures(st["order"], level)
            dense.append((kept, status, z.gather_columns(st["W_snap"][:, slot], kept, case["group"]),
                          z.gather_rows(st["previous"], kept, case["group"])))
        return dense
    if kind == "select":
        return z.select_levels(**st["db"], coef=st["coef"], budget=st["budget"], n_buckets=case["buckets"])
    return z.search_levels(**st["db"], objective=st["objective"], coef0=st["coef0"], budgets=st["budgets"],
                           n_buckets=case["buckets"], mask=st["mask"], values=st["values"])


def work(case):
    kind = case["kind"]
    if kind == "hessian":
        L, d, N = case["layers"], case["cols"], case["tokens"]
        size = 4 if case["dtype"] == "f32" else 2
        return dict(bytes=L * d * N * size + 4 * L * d * d, flops=L * d * (d + 1) * N)
    if kind == "prune":
        L, r, d, g = case["layers"], case["rows"], case["cols"], case["group"]
        levels = _levels(case)
        nbytes = 4 * L * (r * d * (1 + len(levels)) + d * d + 2 * (d // g))
        flops = float(d) ** 3                                    # Cholesky factor and its inverse, H^-1
        for n in range(levels[-1] + 1, d // g + 1):              # n structures live before the step
            c = (n - 1) * g                                      # columns that remain after it
            flops += g * c * (c + 1) + 2.0 * g * r * c           # symmetric downdate of H^-1, update of W
            flops += 2.0 * r * c if g == 1 else n * (g ** 3 + g * g * r)     # saliencies
        return dict(bytes=nbytes, flops=L * flops)
    if kind == "reshape":
        L, r, levels = case["layers"], case["rows"], [v for v in _levels(case) if v > 0]
        moved = sum(v * case["group"] for v in levels) * r * 2   # columns of W, rows of the layer before
        return dict(bytes=L * (8 * moved + 4 * (case["cols"] // case["group"]) + 4 * sum(levels)), flops=0)
    M = case["modules"]
    options = M // 2 * 13 + (M - M // 2) * (1 + len(_paper_sizes(3072)))
    evaluations = 2.0 * options * case["buckets"]                # one addition, one comparison each
    if kind == "select":
        return dict(bytes=8 * options + case["candidates"] * (8 * M + 20), flops=case["candidates"] * evaluations)
    S, T = case["targets"], case["steps"]
    return dict(bytes=12 * options + S * (5 * T * M + 12 * M + 24), flops=S * (T + 1) * evaluations)


def tolerance(case):
    if case["kind"] == "hessian":
        return dict(rel=1e-5)                # sums of fp32 products
    if case["kind"] == "prune":
        # fp32 state over thousands of downdates; two structures may tie to the last digits
        return dict(rel=5e-4, max=2e-2, differ=0.01) if case["group"] == 1 else dict(rel=1e-5)
    return "exact"                           # copies, and float64 sums in a stated order
