"""The work this framework is used for, as cases that can be timed and compared.

Every case calls the public entry points as a serving or training program
does: inputs, weights (folded or prepared once), workspaces and output buffers
are in hand, and one pass is the calls themselves.  Six kinds:

* ``forward``   images to logits: patch embedding, blocks with deletions at
                ``prune_blocks``, classifier (the whole online forward);
* ``block``     one block of a pruned forward, with or without a deletion;
* ``actor``     the deletion decisions of one block from its keys;
* ``embed``     the patch embedding alone;
* ``head``      the classifier on a pruned batch (CLS or LC1 readout);
* ``policy``    the device work of one training rollout action: ordered
                sampling, log-probability with its gradient, shadow branching,
                fidelity costs and local rewards.

Widths, depths, token counts and batch sizes are those of the repository's
workloads (DeiT-Tiny, -Small and -Base, ViT-L, ViT-B/384, DINOv2-B/14);
``draw`` spreads them over the ranges between.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_2609_34325_gb300 as P

BF16, F32, I32, F64 = torch.bfloat16, torch.float32, torch.int32, torch.float64
EPS = 1e-6            # the backbone's LayerNorm epsilon
ACTOR_EPS = 1e-5      # the actor's
CLASSES = 1000        # rows of the classifier, padded to a multiple of the library's 32
CLASSES_PAD = 1024
MAX_ROWS = 50432      # 256 images of 197 tokens: the largest packed batch listed


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one image through a DeiT-Tiny: latency, about a hundred small launches
        {"name": "forward_tiny_1", "kind": "forward", "batch": 1, "dim": 192, "depth": 12,
         "grid": 14, "patch": 16, "lc1": False, "layerscale": False, "prune_blocks": "3,6,9"},
        # the headline workload, images to logits: DeiT-B, 256 images, three deletions
        {"name": "forward_base_256", "kind": "forward", "batch": 256, "dim": 768, "depth": 12,
         "grid": 14, "patch": 16, "lc1": False, "layerscale": False, "prune_blocks": "3,6,9"},
        # a small batch of DeiT-Tiny at a pruning block: an online server's burst
        {"name": "block_tiny_8", "kind": "block", "batch": 8, "tokens": 197, "dim": 192,
         "prune": True, "ragged": False, "layerscale": False},
        # DeiT-Small at a pruning block, a medium batch
        {"name": "block_small_64", "kind": "block", "batch": 64, "tokens": 197, "dim": 384,
         "prune": True, "ragged": False, "layerscale": False},
        # DeiT-Base before its first deletion: most blocks of the headline forward
        {"name": "block_base_256", "kind": "block", "batch": 256, "tokens": 197, "dim": 768,
         "prune": False, "ragged": False, "layerscale": False},
        # ViT-L at a late pruning block: images of very different lengths
        {"name": "block_large_128", "kind": "block", "batch": 128, "tokens": 197, "dim": 1024,
         "prune": True, "ragged": True, "layerscale": False},
        # ViT-B at 384 pixels: long sequences, attention is a quarter of the block
        {"name": "block_base384_64", "kind": "block", "batch": 64, "tokens": 577, "dim": 768,
         "prune": True, "ragged": False, "layerscale": False},
        # DINOv2-B/14 before its first deletion: LayerScale, 257 tokens
        {"name": "block_dino_128", "kind": "block", "batch": 128, "tokens": 257, "dim": 768,
         "prune": False, "ragged": False, "layerscale": True},
        # the actor at the headline forward's first pruning block
        {"name": "actor_base_256", "kind": "actor", "batch": 256, "tokens": 197, "dim": 768,
         "depth": 12, "ragged": False},
        # DINOv2's 14-pixel patches (28-byte pieces of image rows, K = 588)
        {"name": "embed_dino_128", "kind": "embed", "batch": 128, "grid": 16, "patch": 14,
         "dim": 768},
        # DINOv2's LC1 readout after its deletions: every surviving row is read
        {"name": "head_lc1_256", "kind": "head", "batch": 256, "tokens": 143, "dim": 768,
         "lc1": True},
        # a training rollout's policy and shadow work at the first pruning block
        {"name": "policy_base_256", "kind": "policy", "batch": 256, "tokens": 197, "dim": 768},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["forward", "block", "block", "block", "block", "actor", "embed", "head",
                       "policy"])
    if kind == "forward":
        dim = rng.choice([192, 384, 768])
        patch = rng.choice([14, 16])
        grid = rng.randint(8, 24)
        dino = patch == 14
        cap = 30000000 // (dim * (grid * grid + 1))
        return {"kind": "forward", "batch": _log_int(rng, 1, max(1, min(256, cap))), "dim": dim,
                "depth": 12, "grid": grid, "patch": patch, "lc1": dino, "layerscale": dino,
                "prune_blocks": "1,2,3,6" if dino else "3,6,9"}
    if kind == "block":
        tokens = rng.choice([197, 257, 577, _log_int(rng, 17, 577)])
        batch = _log_int(rng, 1, min(512, MAX_ROWS // tokens))
        return {"kind": "block", "batch": batch, "tokens": tokens,
                "dim": rng.choice([192, 384, 768, 1024]), "prune": rng.random() < 0.5,
                "ragged": rng.random() < 0.5, "layerscale": rng.random() < 0.25}
    if kind == "actor":
        grid = rng.choice([14, 16, 24, rng.randint(6, 24)])
        tokens = grid * grid + 1
        return {"kind": "actor", "batch": _log_int(rng, 1, min(512, MAX_ROWS // tokens)),
                "tokens": tokens, "dim": rng.choice([192, 384, 768, 1024]),
                "depth": rng.choice([12, 24]), "ragged": rng.random() < 0.5}
    if kind == "embed":
        grid = rng.randint(6, 24)
        return {"kind": "embed", "batch": _log_int(rng, 1, min(512, MAX_ROWS // (grid * grid))),
                "grid": grid, "patch": rng.choice([14, 16]),
                "dim": rng.choice([192, 384, 768, 1024])}
    tokens = _log_int(rng, 9, 577)
    batch = _log_int(rng, 1, min(1024, MAX_ROWS // tokens))
    dim = rng.choice([192, 384, 768, 1024])
    if kind == "head":
        return {"kind": "head", "batch": batch, "tokens": tokens, "dim": dim,
                "lc1": rng.random() < 0.5}
    return {"kind": "policy", "batch": batch, "tokens": tokens, "dim": dim}


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------

class _Rng:
    """Device draws of one seeded generator, and host draws of another."""

    def __init__(self, seed):
        self.dev = torch.device("cuda:0")
        self.gen = torch.Generator(device=self.dev).manual_seed(seed)
        self.host = torch.Generator().manual_seed(seed ^ 0x5DEECE66D)

    def normal(self, *shape, std=1.0, mean=0.0, dtype=BF16):
        return torch.empty(shape, dtype=F32, device=self.dev).normal_(
            mean, std, generator=self.gen).to(dtype)

    def uniform(self, *shape, lo=0.0, hi=1.0, dtype=F32):
        return torch.empty(shape, dtype=F32, device=self.dev).uniform_(
            lo, hi, generator=self.gen).to(dtype)

    def host_uniform(self, n):
        return torch.rand(n, generator=self.host, dtype=F64)

    def put(self, t, dtype=I32):
        return t.to(dtype).to(self.dev)


def _schedule(case):
    """Rows per image (CLS included) before the first deletion and after each.

    The counts are the same for every seed, which deals them out to the images
    in another order: what is packed has the same size whatever the inputs.
    Ragged images are what an earlier deletion left; a deletion removes an even
    number of rows, 5 to 60 percent, and leaves at least four visual ones."""
    gen = torch.Generator().manual_seed(case["batch"])
    b = case["batch"]
    tokens = case["grid"] ** 2 + 1 if case["kind"] == "forward" else case["tokens"]
    n = torch.full((b,), tokens, dtype=torch.int64)
    if case.get("ragged", case["kind"] == "head"):
        left = 0.2 + 0.8 * torch.rand(b, generator=gen, dtype=F64)
        n = (tokens * left).long().clamp_(min(tokens, 5), tokens)
    counts = [n]
    for _ in range(len(_prune_blocks(case)) if case["kind"] == "forward" else 1):
        f = 0.05 + 0.55 * torch.rand(b, generator=gen, dtype=F64)
        k = 2 * torch.floor(f * (n - 1) / 2 + 0.5).long()
        n = n - torch.minimum(k, (n - 5).clamp_(min=0))
        counts.append(n)
    return counts


def _cu(n):
    return torch.cat([torch.zeros(1, dtype=torch.int64), n.cumsum(0)])


def _block_weights(r, dim, layerscale):
    """One trained-like block: attention logits of a few units, every affine term in play."""
    mlp = 4 * dim
    s = 1.0 / math.sqrt(dim)
    w = {"w_qkv": r.normal(3 * dim, dim, std=1.2 * s), "w_proj": r.normal(dim, dim, std=0.5 * s),
         "w_fc1": r.normal(mlp, dim, std=s), "w_fc2": r.normal(dim, mlp, std=0.5 * s)}
    for name, size in (("b_qkv", 3 * dim), ("b_proj", dim), ("b_fc1", mlp), ("b_fc2", dim),
                       ("ln1_b", dim), ("ln2_b", dim)):
        w[name] = r.normal(size, std=0.1)
    for name in ("ln1_w", "ln2_w"):
        w[name] = r.normal(dim, std=0.1, mean=1.0)
    if layerscale:
        for name in ("ls1", "ls2"):
            w[name] = r.uniform(dim, lo=0.05, hi=0.5, dtype=BF16)
    return w


def _embed_weights(r, dim, patch, grid):
    k = 3 * patch * patch
    return {"w_pe": r.normal(dim, k, std=1.0 / math.sqrt(k)), "b_pe": r.normal(dim, std=0.1),
            "cls": r.normal(dim, std=0.1), "pos": r.normal(grid * grid + 1, dim, std=0.1)}


def _head_weights(r, dim, lc1):
    width = 2 * dim if lc1 else dim
    w = r.normal(CLASSES_PAD, width, std=1.0 / math.sqrt(width))
    b = r.normal(CLASSES_PAD, std=0.1)
    w[CLASSES:] = 0
    b[CLASSES:] = 0
    return {"norm_w": r.normal(dim, std=0.1, mean=1.0), "norm_b": r.normal(dim, std=0.1),
            "w_head": w, "b_head": b}


def _rows(r, rows, dim):
    """A residual stream: per-channel offsets and scales as trained blocks leave them."""
    scale = r.uniform(1, dim, lo=0.5, hi=1.5)
    offset = r.normal(1, dim, std=0.2, dtype=F32)
    return (r.normal(rows, dim, dtype=F32) * scale + offset).to(BF16)


def _actor_weights(r, dim, depth, n0):
    """An actor whose budget head prefers some budgets clearly (a trained head
    does), so that the integer decisions do not hang on the last bit."""
    m = (n0 - 4) // 2

    def mat(out, k, gain=1.0):
        return r.normal(out, k, std=gain / math.sqrt(k))

    def vec(n, mean=0.0):
        return r.normal(n, std=0.1, mean=mean)

    order = torch.randperm(m, generator=r.host)
    return {
        "gate_w1": mat(64, dim + 19), "gate_b1": vec(64), "gate_w2": mat(1, 64, 4.0),
        "gate_b2": vec(1, 0.5), "gate_emb": r.normal(depth, 16, std=0.1),
        "enc_w_in": mat(128, dim), "enc_b_in": vec(128), "enc_emb": r.normal(depth, 128, std=0.1),
        "enc_w_h": mat(128, 3), "enc_ln1_w": vec(128, 1.0), "enc_ln1_b": vec(128),
        "enc_w_qkv": mat(384, 128), "enc_b_qkv": vec(384), "enc_w_o": mat(128, 128),
        "enc_b_o": vec(128), "enc_ln2_w": vec(128, 1.0), "enc_ln2_b": vec(128),
        "enc_w_fc1": mat(256, 128), "enc_b_fc1": vec(256), "enc_w_fc2": mat(128, 256),
        "enc_b_fc2": vec(128), "bud_ln_w": vec(128, 1.0), "bud_ln_b": vec(128),
        "bud_w1": mat(128, 128), "bud_b1": vec(128), "bud_w2": mat(m, 128, 0.1),
        "bud_b2": r.put(0.5 * (order - m // 2).double(), BF16), "sel_w_k": vec(128),
        "sel_w1": mat(64, 128), "sel_b1": vec(64), "sel_w2": mat(1, 64), "sel_b2": vec(1),
    }


def _inputs(case, seed):
    """Everything drawn for a case: device tensors, and host lists of lengths and keep counts."""
    r = _Rng(seed)
    kind, b, dim = case["kind"], case["batch"], case["dim"]
    i = {}
    if kind in ("forward", "embed"):
        side = case["grid"] * case["patch"]
        i["images"] = r.normal(b, 3, side, side)
        i["embed"] = _embed_weights(r, dim, case["patch"], case["grid"])
    if kind == "embed":
        return i
    order = torch.randperm(b, generator=r.host)
    counts = [n[order] for n in _schedule(case)]
    n, i["n"] = counts[0], counts[0]
    if kind == "forward":
        i["blocks"] = [_block_weights(r, dim, case["layerscale"]) for _ in range(case["depth"])]
        i["head"] = _head_weights(r, dim, case["lc1"])
        i["prune"] = {l: (m, r.uniform(b, case["grid"] ** 2 + 1))
                      for l, m in zip(_prune_blocks(case), counts[1:])}
        return i
    rows = int(n.sum())
    i["cu"] = r.put(_cu(n))
    if kind == "block":
        i["x"] = _rows(r, rows, dim)
        i["weights"] = _block_weights(r, dim, case["layerscale"])
        # original token ids: a sorted subset of each image's tokens where some are gone
        i["ids"] = r.put(torch.cat([torch.cat([torch.zeros(1, dtype=torch.int64), 1 + torch.randperm(
            case["tokens"] - 1, generator=r.host)[:int(v) - 1].sort().values]) for v in n]))
        if case["prune"]:
            i["keep"], i["scores"] = counts[1], r.uniform(rows)
    elif kind == "actor":
        i["qkv"] = r.normal(rows, 3 * dim)
        i["weights"] = _actor_weights(r, dim, case["depth"], case["tokens"] - 1)
        i["rho"] = r.put(0.4 * r.host_uniform(b), F32)
        i["interventions"] = r.put(torch.floor(3 * r.host_uniform(b)))
    elif kind == "head":
        i["x"] = _rows(r, rows, dim)
        i["head"] = _head_weights(r, dim, case["lc1"])
    else:
        u = r.uniform(rows).clamp_(1e-7, 1 - 1e-6)
        i["scores"], i["gumbel"] = r.normal(rows, dtype=F32), -torch.log(-torch.log(u))
        i["k"] = n - counts[1]
        i["dlogp"] = r.normal(b, dtype=F32)
        i["x"], i["mv"] = _rows(r, rows, dim), r.uniform(rows, 2, lo=0.1)
        i["logits"] = r.normal(3 * b, CLASSES_PAD, std=3.0)     # rollout, Native, one shadow group
    return i


def _prune_blocks(case):
    return [int(v) for v in case["prune_blocks"].split(",")]


# ---------------------------------------------------------------------------
# what a program keeps, and one pass
# ---------------------------------------------------------------------------

def _zeros(*shape, dtype=BF16):
    return torch.zeros(shape, dtype=dtype, device="cuda:0")


def prepare(case, seed):
    i = _inputs(case, seed)
    kind, b, dim = case["kind"], case["batch"], case["dim"]
    s = {"kind": kind, "case": case, "i": i}
    if kind in ("forward", "embed"):
        s["x0"] = _zeros(b * (case["grid"] ** 2 + 1), dim)
        e = i["embed"]
        s["embed_ws"] = P.dora_patch_embed(i["images"], e["w_pe"], e["b_pe"], e["cls"], e["pos"],
                                           case["patch"], s["x0"])
    if kind in ("forward", "head"):
        head = P.dora_classifier_head_lc1 if case["lc1"] else P.dora_classifier_head
        h = i["head"]
        s["logits"] = _zeros(b, CLASSES_PAD)
        cu = i["cu"] if kind == "head" else _cu(i["n"]).to(I32).cuda()
        x = i["x"] if kind == "head" else s["x0"]
        s["head"], s["head_ws"] = head, head(x, cu, h["norm_w"], h["norm_b"], EPS, h["w_head"],
                                             h["b_head"], s["logits"])
    if kind == "forward":
        tokens, rows = case["grid"] ** 2 + 1, b * (case["grid"] ** 2 + 1)
        s["blocks"] = [P.BlockWeights(w, dim, dim // 64, 4 * dim, EPS).fold() for w in i["blocks"]]
        s["ws"] = P.alloc_workspace(rows, b, s["blocks"][0])
        s["x"] = [s["x0"], _zeros(rows, dim), _zeros(rows, dim)]
        s["mv"] = [_zeros(rows, 2, dtype=F32) for _ in range(2)]
        s["cu"] = [_cu(i["n"]).to(I32).cuda()] + [_zeros(b + 1, dtype=I32) for _ in i["prune"]]
        s["ids"] = [torch.arange(tokens, dtype=I32, device="cuda:0").repeat(b)] + [
            _zeros(rows, dtype=I32) for _ in i["prune"]]
        s["keep"] = {l: n.to(I32).cuda() for l, (n, _) in i["prune"].items()}
        s["scores"], s["status"] = _zeros(rows, dtype=F32), _zeros(1, dtype=I32)
        s["rows_out"] = int(list(i["prune"].values())[-1][0].sum())
    elif kind == "block":
        rows = i["x"].shape[0]
        s["w"] = P.BlockWeights(i["weights"], dim, dim // 64, 4 * dim, EPS).fold()
        s["ws"] = P.alloc_workspace(rows, b, s["w"])
        s["mv_in"], s["mv_out"] = _zeros(rows, 2, dtype=F32), _zeros(rows, 2, dtype=F32)
        P.dora_row_stats(i["x"], s["mv_in"])                 # what the block before hands over
        s["x_out"] = _zeros(rows, dim)
        s["rows_out"] = rows
        if case["prune"]:
            s["keep"] = i["keep"].to(I32).cuda()
            s["cu_out"] = _zeros(b + 1, dtype=I32)
            s["ids_out"], s["kept"] = _zeros(rows, dtype=I32), _zeros(rows, dtype=I32)
            s["rows_out"] = int(i["keep"].sum())
    elif kind == "actor":
        rows = i["qkv"].shape[0]
        s["w"] = P.ActorWeights(i["weights"], dim, case["depth"], case["tokens"] - 1,
                                ACTOR_EPS).prepare()
        s["ws"] = P.alloc_actor_workspace(rows, b, s["w"])
        s["out"] = {name: _zeros(b, dtype=I32)
                    for name in ("gate", "budget", "k", "keep_counts", "interventions_next")}
        s["out"].update({name: _zeros(b, dtype=F32) for name in ("p_gate", "rho_next")})
        s["out"]["scores"], s["out"]["z_out"] = _zeros(rows, dtype=F32), _zeros(rows, 128)
    elif kind == "policy":
        rows, k_cap = i["x"].shape[0], case["tokens"] - 1
        s["x"] = torch.cat([i["x"], _zeros(rows, dim)])      # room for the shadows
        s["mv"] = torch.cat([i["mv"], _zeros(rows, 2, dtype=F32)])
        s["ids"] = torch.arange(2 * rows, dtype=I32, device="cuda:0")
        s["src"] = torch.arange(b, dtype=I32, device="cuda:0")
        s["k"] = i["k"].to(I32).cuda()
        s["cu_out"], s["len"] = _zeros(2 * b + 1, dtype=I32), _zeros(b, dtype=I32)
        s["order"] = _zeros(b, k_cap, dtype=I32)
        s["keys"], s["grad"] = _zeros(rows, dtype=F32), _zeros(rows, dtype=F32)
        s["logp"], s["cost"] = _zeros(b, dtype=F32), _zeros(3 * b, dtype=F32)
        s["image_of"] = torch.arange(3 * b, dtype=I32, device="cuda:0") % b
        s["removals"] = torch.stack([s["k"], s["k"] // 2])
        s["blocks"] = torch.tensor([3, 6], dtype=I32, device="cuda:0")
        s["reward"], s["ret"] = _zeros(2, b, dtype=F32), _zeros(b, dtype=F32)
    return s


def _run_forward(s):
    i, case = s["i"], s["case"]
    e, h = i["embed"], i["head"]
    P.dora_patch_embed(i["images"], e["w_pe"], e["b_pe"], e["cls"], e["pos"], case["patch"],
                       s["x0"], s["embed_ws"])
    tokens, depth = case["grid"] ** 2 + 1, case["depth"]
    x, mv, at = s["x0"], None, 0
    for l, w in enumerate(s["blocks"]):
        out = s["x"][1 + l % 2]
        mv_out = s["mv"][l % 2] if l + 1 < depth else None
        if l in s["keep"]:
            P.dora_gather_scores(i["prune"][l][1], s["ids"][at], s["cu"][at], s["scores"],
                                 status=s["status"])
            P.dora_pruned_block(x, s["cu"][at], w, tokens, out, s["ws"], ids_in=s["ids"][at],
                                scores=s["scores"], keep_counts=s["keep"][l],
                                cu_out=s["cu"][at + 1], ids_out=s["ids"][at + 1],
                                x_in_moments=mv, x_out_moments=mv_out)
            at += 1
        else:
            P.dora_pruned_block(x, s["cu"][at], w, tokens, out, s["ws"], x_in_moments=mv,
                                x_out_moments=mv_out)
        x, mv = out, mv_out
    s["head"](x, s["cu"][at], h["norm_w"], h["norm_b"], EPS, h["w_head"], h["b_head"],
              s["logits"], s["head_ws"])
    # the surviving tokens' features and the logits; rows past the survivors are room
    n = s["rows_out"]
    return {"logits": s["logits"], "x": x[:n], "cu": s["cu"][at], "ids": s["ids"][at][:n]}


def run(state):
    s, i, case = state, state["i"], state["case"]
    kind = s["kind"]
    if kind == "forward":
        return _run_forward(s)
    if kind == "block":
        n = s["rows_out"]
        if not case["prune"]:
            P.dora_pruned_block(i["x"], i["cu"], s["w"], case["tokens"], s["x_out"], s["ws"],
                                x_in_moments=s["mv_in"], x_out_moments=s["mv_out"])
            return {"x_out": s["x_out"], "moments": s["mv_out"]}
        P.dora_pruned_block(i["x"], i["cu"], s["w"], case["tokens"], s["x_out"], s["ws"],
                            ids_in=i["ids"], scores=i["scores"], keep_counts=s["keep"],
                            cu_out=s["cu_out"], ids_out=s["ids_out"], kept_idx=s["kept"],
                            x_in_moments=s["mv_in"], x_out_moments=s["mv_out"])
        # rows past the survivors are room, not results
        return {"x_out": s["x_out"][:n], "moments": s["mv_out"][:n], "cu": s["cu_out"],
                "ids": s["ids_out"][:n], "kept": s["kept"][:n]}
    if kind == "actor":
        P.dora_actor(i["qkv"], i["cu"], s["w"], 3, case["tokens"], i["rho"], i["interventions"],
                     workspace=s["ws"], **s["out"])
        return s["out"]
    if kind == "embed":
        e = i["embed"]
        P.dora_patch_embed(i["images"], e["w_pe"], e["b_pe"], e["cls"], e["pos"], case["patch"],
                           s["x0"], s["embed_ws"])
        return s["x0"]
    if kind == "head":
        h = i["head"]
        s["head"](i["x"], i["cu"], h["norm_w"], h["norm_b"], EPS, h["w_head"], h["b_head"],
                  s["logits"], s["head_ws"])
        return s["logits"]
    b = case["batch"]
    P.dora_pl_sample(i["scores"], i["gumbel"], i["cu"], s["k"], s["order"], keys_out=s["keys"])
    P.dora_pl_logprob(i["scores"], i["cu"], s["k"], s["order"], s["logp"], grad=s["grad"],
                      dlogp=i["dlogp"])
    P.dora_branch(s["x"], i["cu"], s["src"], s["cu_out"], ids=s["ids"], x_moments=s["mv"],
                  len_out=s["len"])
    P.dora_kd_cost(i["logits"][b:2 * b], i["logits"], s["cost"], CLASSES,
                   shadow_image=s["image_of"])
    P.dora_step_rewards(s["cost"], s["removals"], s["blocks"], 12, case["tokens"] - 1, 1.0,
                        s["reward"], ret=s["ret"])
    return {"order": s["order"], "keys": s["keys"], "logp": s["logp"], "grad": s["grad"],
            "x": s["x"], "ids": s["ids"], "mv": s["mv"], "cu": s["cu_out"], "len": s["len"],
            "cost": s["cost"], "reward": s["reward"], "ret": s["ret"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _block_work(n_in, n_out, dim):
    """(bytes, flops) of one block: rows and weights once, attention per image."""
    t_in, t_out = float(n_in.sum()), float(n_out.sum())
    flops = 2 * t_in * dim * 4 * dim + 2 * t_out * dim * 8 * dim + 4 * float((n_in ** 2).sum()) * dim
    return 2 * dim * (t_in + t_out) + 2 * 12 * dim * dim, flops


def _embed_work(case):
    k, g, dim = 3 * case["patch"] ** 2, case["grid"] ** 2, case["dim"]
    b = case["batch"]
    return 2 * (b * g * k + dim * k + b * (g + 1) * dim + (g + 1) * dim), 2 * b * g * k * dim


def work(case):
    kind, b, dim = case["kind"], case["batch"], case["dim"]
    if kind == "embed":
        nbytes, flops = _embed_work(case)
        return {"bytes": nbytes, "flops": flops}
    counts = _schedule(case)
    if kind == "forward":
        nbytes, flops = _embed_work(case)
        nbytes -= 2 * b * (case["grid"] ** 2 + 1) * dim          # the tokens stay inside the pass
        left = iter(counts[1:])
        n = counts[0]
        for l in range(case["depth"]):
            m = next(left) if l in _prune_blocks(case) else n
            f = _block_work(n, m, dim)[1]
            nbytes, flops, n = nbytes + 2 * 12 * dim * dim, flops + f, m
        width = 2 * dim if case["lc1"] else dim
        return {"bytes": nbytes + 2 * CLASSES_PAD * (width + b),
                "flops": flops + 2 * b * CLASSES_PAD * width}
    n = counts[0]
    t = float(n.sum())
    if kind == "block":
        m = counts[1] if case["prune"] else n
        nbytes, flops = _block_work(n, m, dim)
        extra = 8 * (t + float(m.sum())) + (8 * t + 8 * float(m.sum()) if case["prune"] else 0)
        return {"bytes": nbytes + extra, "flops": flops}
    if kind == "actor":
        # keys in, z and scores out; the encoder's, selector's and gate's products
        per_row = 2 * 128 * (dim + 3 * 128 + 128 + 2 * 256 + 64)
        flops = t * per_row + 4 * float((n ** 2).sum()) * 128 + 2 * b * 64 * (dim + 19)
        return {"bytes": t * (2 * dim + 2 * 128 + 4), "flops": flops}
    if kind == "head":
        width = 2 * dim if case["lc1"] else dim
        rows = t if case["lc1"] else b
        return {"bytes": 2 * (rows * dim + CLASSES_PAD * width + b * CLASSES_PAD),
                "flops": 2 * b * CLASSES_PAD * width}
    per_row = 4 * 3 + 4 * 2 + 2 * (2 * dim + 8 + 4)              # scores, keys, grad; the copies
    return {"bytes": t * per_row + 4 * b * case["tokens"] + 2 * 3 * b * CLASSES, "flops": 0}


# ---------------------------------------------------------------------------
# tolerances and the 64-bit results
# ---------------------------------------------------------------------------

def tolerance(case):
    # bf16 results of bf16 inputs with 32-bit sums inside: about four times what the
    # outputs are from exact(); a forward is its twelve blocks' roundings together
    return {"forward": {"rel": 0.03}, "block": {"rel": 0.01}, "actor": {"rel": 0.015},
            "embed": {"rel": 0.01}, "head": {"rel": 0.01}, "policy": {"rel": 1e-5}}[case["kind"]]


def _d(t):
    return t.to(F64)


def _ln(x, w, b, eps):
    return F.layer_norm(x, (x.shape[-1],), _d(w), _d(b), eps)


def _lin(x, w, b):
    return x @ _d(w).T + _d(b)


def _attention(qkv, n, heads, scale):
    """softmax(Q K^T scale) V within each image, rows packed image after image."""
    rows, width = qkv.shape
    hd = width // (3 * heads)
    longest = int(n.max())
    out = torch.empty(rows, heads * hd, dtype=F64, device=qkv.device)
    lo = _cu(n).tolist()
    step = max(1, int(4e8 // (heads * longest * longest)))
    for a in range(0, n.numel(), step):
        part = n[a:a + step]
        live = (torch.arange(longest) < part[:, None]).to(qkv.device)
        pad = torch.zeros(part.numel(), longest, width, dtype=F64, device=qkv.device)
        pad[live] = qkv[lo[a]:lo[a + part.numel()]]
        q, k, v = pad.view(part.numel(), longest, 3, heads, hd).permute(2, 0, 3, 1, 4)
        logits = (q @ k.transpose(-1, -2)) * scale
        p = logits.masked_fill_(~live[:, None, None, :], -math.inf).softmax(-1)
        out[lo[a]:lo[a + part.numel()]] = (p @ v).transpose(1, 2).reshape(
            part.numel(), longest, heads * hd)[live]
    return out


def _select(scores, n, keep):
    """Rows kept: CLS and the lowest scores, ties to the lower index, in order."""
    longest = int(n.max())
    live = torch.arange(longest) < n[:, None]
    pad = torch.full((n.numel(), longest), math.inf, dtype=F32)
    pad[live] = scores.cpu()
    pad[:, 0] = -math.inf
    rank = pad.sort(dim=1, stable=True).indices.argsort(dim=1)
    return torch.nonzero((rank < keep[:, None])[live]).squeeze(1)


def _exact_block(x, w, n, heads, scores=None, keep=None):
    """Eq. 1 on rows in 64 bits: (rows out, kept row indices or None)."""
    qkv = _lin(_ln(x, w["ln1_w"], w["ln1_b"], EPS), w["w_qkv"], w["b_qkv"])
    branch = _lin(_attention(qkv, n, heads, 0.125), w["w_proj"], w["b_proj"])
    x = x + (branch * _d(w["ls1"]) if "ls1" in w else branch)
    kept = None
    if scores is not None:
        kept = _select(scores, n, keep).to(x.device)
        x = x[kept]
    hidden = F.gelu(_lin(_ln(x, w["ln2_w"], w["ln2_b"], EPS), w["w_fc1"], w["b_fc1"]))
    branch = _lin(hidden, w["w_fc2"], w["b_fc2"])
    return x + (branch * _d(w["ls2"]) if "ls2" in w else branch), kept


def _exact_embed(images, e, patch):
    b, _, h, w = images.shape
    emb = F.unfold(_d(images), patch, stride=patch).transpose(1, 2) @ _d(e["w_pe"]).T + _d(e["b_pe"])
    cls = _d(e["cls"]).expand(b, 1, -1)
    return (torch.cat([cls, emb], 1) + _d(e["pos"])).reshape(-1, emb.shape[-1])


def _exact_head(x, n, h, lc1):
    lo = _cu(n)[:-1].to(x.device)
    feat = _ln(x[lo], h["norm_w"], h["norm_b"], EPS)
    if lc1:
        y = _ln(x, h["norm_w"], h["norm_b"], EPS)
        image = torch.repeat_interleave(torch.arange(n.numel()), n).to(x.device)
        total = torch.zeros_like(feat).index_add_(0, image, y) - y[lo]
        feat = torch.cat([feat, total / (n - 1).clamp(min=1)[:, None].to(x.device)], 1)
    return _lin(feat, h["w_head"], h["b_head"])


def _exact_actor(case, i):
    w, n, dim = i["weights"], i["n"], case["dim"]
    n0, block, vis = case["tokens"] - 1, 3, (i["n"] - 1).cuda()
    lo = _cu(n)[:-1].cuda()
    keys = _d(i["qkv"][:, dim:2 * dim])
    h = torch.stack([vis.double() / n0, _d(i["rho"]),
                     _d(i["interventions"]) / max(case["depth"] - 1, 1)], 1)
    z = torch.cat([keys[lo], _d(w["gate_emb"])[block].expand(n.numel(), -1), h], 1)
    p = torch.sigmoid(_lin(F.silu(_lin(z, w["gate_w1"], w["gate_b1"])), w["gate_w2"],
                           w["gate_b2"]))[:, 0]
    x = _lin(keys, w["enc_w_in"], w["enc_b_in"]) + _d(w["enc_emb"])[block]
    x[lo] += h @ _d(w["enc_w_h"]).T
    qkv = _lin(_ln(x, w["enc_ln1_w"], w["enc_ln1_b"], ACTOR_EPS), w["enc_w_qkv"], w["enc_b_qkv"])
    x = x + _lin(_attention(qkv, n, 4, 32 ** -0.5), w["enc_w_o"], w["enc_b_o"])
    f = F.gelu(_lin(_ln(x, w["enc_ln2_w"], w["enc_ln2_b"], ACTOR_EPS), w["enc_w_fc1"],
                    w["enc_b_fc1"]))
    z = x + _lin(f, w["enc_w_fc2"], w["enc_b_fc2"])
    u = F.gelu(_lin(_ln(z[lo], w["bud_ln_w"], w["bud_ln_b"], ACTOR_EPS), w["bud_w1"], w["bud_b1"]))
    logits = _lin(u, w["bud_w2"], w["bud_b2"])
    grid = torch.arange(2, n0 - 3, 2, device=x.device)[:logits.shape[1]]
    feasible = grid <= (vis - 4)[:, None]
    best = grid[logits.masked_fill(~feasible, -math.inf).argmax(1)]
    budget = torch.where(feasible.any(1), best, torch.zeros_like(best))
    gate = ((p >= 0.5) & (budget > 0)).long()
    k = budget * gate
    image = torch.repeat_interleave(torch.arange(n.numel()), n).cuda()
    ratio = (budget / vis.clamp(min=1))[image][:, None]
    scores = _lin(F.silu(_lin(z + ratio * _d(w["sel_w_k"]), w["sel_w1"], w["sel_b1"])),
                  w["sel_w2"], w["sel_b2"])[:, 0]
    scores[lo] = 0
    return {"gate": gate, "budget": budget, "k": k, "keep_counts": n.cuda() - k,
            "interventions_next": i["interventions"] + gate, "p_gate": p,
            "rho_next": k / vis.clamp(min=1).double(), "scores": scores, "z_out": z}


def _exact_policy(case, i):
    b, n = case["batch"], i["n"]
    lo = _cu(n).tolist()
    scores, keys = _d(i["scores"]).cpu(), (i["scores"] + i["gumbel"]).cpu()
    keys[_cu(n)[:-1]] = i["scores"].cpu()[_cu(n)[:-1]]
    order = torch.full((b, case["tokens"] - 1), -1, dtype=torch.int64)
    grad, logp, dlogp = torch.zeros_like(scores), torch.zeros(b, dtype=F64), i["dlogp"].cpu()
    for a in range(b):
        k = int(i["k"][a])
        key, s = keys[lo[a] + 1:lo[a + 1]], scores[lo[a] + 1:lo[a + 1]]
        # the largest keys first, ties to the higher index
        seq = (key.numel() - 1 - key.flip(0).sort(descending=True, stable=True).indices)[:k]
        order[a, :k] = seq
        if k == 0:
            continue
        rest = torch.ones_like(s, dtype=torch.bool)
        rest[seq] = False
        base = torch.logsumexp(s[rest], 0).expand(1)
        left = torch.logcumsumexp(torch.cat([base, s[seq].flip(0)]), 0)[1:].flip(0)
        logp[a] = (s[seq] - left).sum()
        prefix = torch.logcumsumexp(-left, 0)
        g = -torch.exp(s + prefix[-1])
        g[seq] = 1 - torch.exp(s[seq] + prefix)
        grad[lo[a] + 1:lo[a + 1]] = g * dlogp[a]
    z = _d(i["logits"][:, :CLASSES]) / 3.0
    native = z[b:2 * b].log_softmax(1).repeat(3, 1)
    cost = 9.0 * (native.exp() * (native - z.log_softmax(1))).sum(1)
    # branched after the first of two pruning blocks: rollout, Native, one group of shadows
    rollout, shadow = cost[:b], cost[2 * b:]
    k = i["k"].cuda()
    removals = torch.stack([k, k // 2]).double()
    saved = 25.0 * removals * torch.tensor([[9.0], [6.0]], dtype=F64, device=k.device) / (
        12.0 * (case["tokens"] - 1))
    reward = saved - torch.stack([shadow, rollout - shadow])
    rows = i["x"].shape[0]
    ids = torch.arange(rows).repeat(2)
    return {"order": order, "keys": keys.double(), "logp": logp, "grad": grad,
            "x": _d(torch.cat([i["x"], i["x"]])), "ids": ids, "mv": _d(torch.cat([i["mv"], i["mv"]])),
            "cu": torch.cat([_cu(n), lo[-1] + _cu(n)[1:]]), "len": n, "cost": cost,
            "reward": reward, "ret": reward.sum(0)}


def exact(case, seed):
    if work(case)["flops"] > 9e12:          # 64-bit products run at about 1 TFLOP/s
        return None
    i = _inputs(case, seed)
    kind, heads = case["kind"], case["dim"] // 64
    if kind == "embed":
        return _exact_embed(i["images"], i["embed"], case["patch"])
    if kind == "head":
        return _exact_head(_d(i["x"]), i["n"], i["head"], case["lc1"])
    if kind == "actor":
        return _exact_actor(case, i)
    if kind == "policy":
        return _exact_policy(case, i)
    n = i["n"]
    if kind == "block":
        x, kept = _exact_block(_d(i["x"]), i["weights"], n, heads, i.get("scores"), i.get("keep"))
        var, mean = torch.var_mean(x, 1, correction=0)
        out = {"x_out": x, "moments": torch.stack([mean, var], 1)}
        if kept is not None:
            out.update(cu=_cu(i["keep"]), ids=i["ids"][kept], kept=kept)
        return out
    x = _exact_embed(i["images"], i["embed"], case["patch"])
    ids = torch.arange(case["grid"] ** 2 + 1).repeat(case["batch"])
    for l, w in enumerate(i["blocks"]):
        if l in i["prune"]:
            keep, table = i["prune"][l]
            image = torch.repeat_interleave(torch.arange(case["batch"]), n)
            x, kept = _exact_block(x, w, n, heads, table[image.cuda(), ids.cuda()], keep)
            ids, n = ids[kept.cpu()], keep
        else:
            x, _ = _exact_block(x, w, n, heads)
    return {"logits": _exact_head(x, n, i["head"], case["lc1"]), "x": x, "cu": _cu(n), "ids": ids}
