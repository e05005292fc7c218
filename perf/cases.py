"""Performance cases of the AVQ-attention library: what its users have it compute, through the Python binding.

A case names an entry point (``kind``) and a problem:

  forward   ``binding.Forward`` planned once per shape, then called with new Q, K, V (bf16 on the tensor cores,
            fp32 on the CUDA cores; ``stays`` sets the PARENT_STAYS child rule)
  attend    ``Forward.attend``: further queries over keys that an earlier call has already quantised
  permuted  ``binding.forward_permuted``: image tokens tiled along a space-filling curve
  tiled     ``binding.forward_tiled``: codebooks too large to score in one tile
  update    ``binding.codebook_update``: one training-time update of codebooks and EMA statistics

Sizes are those of the repository's configurations (``synth.C0`` .. ``synth.C3``, the N x M x P sweep, the capture
table's large codebooks, the ViT-B and DPT-L sequence lengths 785 and 901).  Inputs follow the recipe of
``paper_2607_12789_b200/synth.py`` (codewords, Dirichlet-weighted clusters of keys, queries around a few hot
parents or spread out), drawn on the GPU because the largest ones take seconds with numpy.
"""
import math

import numpy as np
import torch

from paper_2607_12789_b200 import binding


def _case(kind, B, H, Nq, Nk, d, M, C, P, block_q=128, dtype="bf16", stays=False, hot=True, alpha=0.3, tile_m=0):
    return dict(kind=kind, B=B, H=H, Nq=Nq, Nk=Nk, d=d, M=M, C=C, P=P, block_q=block_q, dtype=dtype, stays=stays,
                hot=hot, alpha=alpha, tile_m=tile_m)


def listed():
    return [
        # the smallest call: one head of the fp32 configuration (launches and latency are all there is)
        dict(_case("forward", 1, 1, 256, 256, 64, 16, 4, 2, block_q=64, dtype="f32", hot=False, alpha=0.0),
             name="tiny_f32"),
        # fp32 inference of a small batch: the precision a user falls back to when checking a bf16 deployment
        dict(_case("forward", 2, 12, 1024, 1024, 64, 64, 4, 8, dtype="f32", hot=False, alpha=0.5), name="batch_f32"),
        # one image through one ViT-B layer: a ragged 785-token sequence, latency-bound
        dict(_case("forward", 1, 12, 785, 785, 64, 64, 4, 8, hot=False, alpha=0.5), name="one_image"),
        # a batch of images (configuration c1)
        dict(_case("forward", 8, 12, 1024, 1024, 64, 64, 4, 8, hot=False, alpha=0.5), name="image_batch"),
        # latent-diffusion self-attention (configuration c2)
        dict(_case("forward", 2, 16, 4096, 4096, 64, 128, 8, 16), name="mid"),
        # long sequence, wide heads (configuration c3)
        dict(_case("forward", 1, 16, 16384, 16384, 128, 256, 4, 32), name="long"),
        # the longest sweep point with its largest codebook
        dict(_case("forward", 1, 16, 65536, 65536, 64, 256, 4, 64), name="longest"),
        # the other child rule (keys may stay with their parent), ragged length, a codebook width between two tiles
        dict(_case("forward", 2, 8, 5000, 5000, 128, 96, 8, 12, stays=True), name="stays_ragged"),
        # queries of another length over keys quantised once (cross-attention, repeated denoising steps)
        dict(_case("attend", 4, 12, 901, 4096, 64, 128, 4, 32), name="attend_cached_keys"),
        # image tokens grouped along a space-filling curve: 64 x 64 latents
        dict(_case("permuted", 2, 16, 4096, 4096, 64, 128, 8, 16), name="curve_order"),
        # a codebook beyond one tile, selection from the tiled importance (capture table: M 512, P 64, tile 128)
        dict(_case("tiled", 1, 4, 4096, 4096, 64, 512, 4, 64, tile_m=128), name="tiled_codebook"),
        # one codebook update of a training step at the mid configuration
        dict(_case("update", 2, 16, 4096, 4096, 64, 128, 8, 16), name="codebook_update"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another call of the same ranges.  Kinds appear as often as they are listed."""
    kind = rng.choice(["forward"] * 6 + ["forward_f32"] * 2 + ["attend", "permuted", "tiled", "update"])
    hot = rng.random() < 0.7
    alpha = rng.choice([0.3, 0.5, 0.8])
    if kind == "forward_f32":
        d = rng.choice([36, 64, 64, 96, 128])
        M = rng.choice([11, 16, 32, 64, 100])
        C = rng.choice([3, 4, 4, 8])
        P = max(1, M // rng.choice([4, 8]))
        block_q = rng.choice([50, 64, 128])
        heads = rng.choice([1, 2, 4, 12])
        N = _log_int(rng, 200, max(400, 2 * 12 * 1024 * 64 * 96 // (heads * d * (M + P * C))))
        N = min(N, 4096)
        return _case("forward", 1, heads, N, N, d, M, C, P, block_q=block_q, dtype="f32", hot=hot, alpha=alpha)
    if kind == "tiled":
        M = rng.choice([512, 768, 1024])
        P = M // rng.choice([8, 16])
        tile_m = rng.choice([128, 256])
        most = 4 * 4096 * (512 + 256) // (M + 4 * P)           # query tokens of all heads
        heads = rng.choice([1, 2, 4])
        N = _log_int(rng, 300, most // heads)
        return _case("tiled", 1, heads, N, N, 64, M, 4, P, tile_m=tile_m, hot=hot, alpha=alpha)
    d = rng.choice([64, 64, 128])
    M = rng.choice([32, 64, 64, 96, 128, 128, 256])
    C = rng.choice([4, 4, 8])
    P = M // rng.choice([4, 8, 8, 16])
    B, H = rng.choice([(1, 12), (1, 16), (2, 16), (4, 12), (8, 12)])
    # tokens of all heads so that neither the flops nor the bytes of the longest listed case are exceeded
    most = 16 * 65536 * min(1.0, (2 * (256 + 4 * 64) + 256) / (2 * (M + P * C) + M + C)) * 64 / d
    N = _log_int(rng, 197, min(65536, int(most) // (B * H) - 1))
    if kind == "attend":
        Nk = _log_int(rng, 512, 8192)
        return _case("attend", B, H, min(N, 8192), Nk, d, M, C, P, hot=hot, alpha=alpha)
    if kind in ("permuted", "update"):
        return _case(kind, B, H, min(N, 16384), min(N, 16384), d, M, C, P, hot=hot, alpha=alpha)
    return _case("forward", B, H, N, N, d, M, C, P, stays=rng.random() < 0.25, hot=hot, alpha=alpha)


# ------------------------------------------------------------------------------------------------ inputs
def _inputs(c, seed, want):
    """Arrays of the synth recipe, drawn on the GPU from the seed alone."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(1_000_003 * seed + 17)
    h = np.random.default_rng(seed)
    B, H, Nq, Nk, d, M, C = (c[k] for k in ("B", "H", "Nq", "Nk", "d", "M", "C"))
    td = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    normal = lambda *s: torch.randn(*s, device=dev, generator=g)
    Cp = (3.0 * normal(H, M, d)).to(td)
    Cc = (Cp.float()[:, :, None, :] + (1.2 if d == 128 else 0.5) * normal(H, M, C, d)).to(td)
    out = dict(Cp=Cp, Cc=Cc)
    if "K" in want:
        pi = np.full((B * H, M), 1.0 / M) if c["alpha"] == 0.0 else h.dirichlet(np.full(M, c["alpha"]), size=B * H)
        pi = torch.from_numpy(pi).to(dev).float()
        pj = torch.multinomial(pi, Nk, replacement=True, generator=g).view(B, H, Nk)
        cj = torch.randint(0, C, (B, H, Nk), device=dev, generator=g)
        head = torch.arange(H, device=dev)[None, :, None]
        K = Cc[head, pj, cj].float() + 0.3 * normal(B, H, Nk, d)
        if c["stays"]:                                          # every other key hugs its parent: it stays with it
            K[:, :, ::2] = Cp[head, pj[:, :, ::2]].float() + 0.05 * normal(B, H, (Nk + 1) // 2, d)
        out["K"] = K.to(td)
    if "V" in want:
        out["V"] = normal(B, H, Nk, d).to(td)
    if "Q" in want:
        Q = normal(B, H, Nq, d)
        if c["hot"]:                                            # around a random tenth of the parents of each (b, h)
            n_hot = max(1, math.ceil(0.1 * M))
            hot = torch.rand(B, H, M, device=dev, generator=g).argsort(-1)[..., :n_hot]
            pick = hot.gather(-1, torch.randint(0, n_hot, (B, H, Nq), device=dev, generator=g))
            Q += Cp[torch.arange(H, device=dev)[None, :, None], pick].float()
        out["Q"] = Q.to(td)
    return out


def _curve(n):
    """Tokens 0..n-1 of a square image in Z-order: the permutation a tile of neighbouring tokens comes from."""
    side = math.isqrt(n - 1) + 1
    i = np.arange(n)
    x, y = i % side, i // side
    key = np.zeros(n, dtype=np.int64)
    for b in range(16):
        key |= ((x >> b) & 1) << (2 * b) | ((y >> b) & 1) << (2 * b + 1)
    return torch.from_numpy(np.argsort(key, kind="stable").astype(np.int32)).cuda()


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    s = dict(c=c)
    if kind == "update":
        s.update(_inputs(c, seed, "K"))
        H, M, C, d = c["H"], c["M"], c["C"], c["d"]
        # statistics of a training run in progress: about as much mass as a batch brings, a few codes never used
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 5)
        rand = lambda *t: torch.rand(*t, device="cuda", generator=g)
        Nc = 2.0 * c["B"] * c["Nk"] / (M * C) * rand(H, M, C)
        Nc[:, ::31, 0] = 0.0
        Sc = Nc[..., None] * s["Cc"].float()
        s["stats"] = [Sc.sum(2).contiguous(), Nc.sum(2).contiguous(), Sc.contiguous(), Nc.contiguous()]
        return s
    s.update(_inputs(c, seed, "QKV"))
    if kind == "permuted":
        s["perm"] = _curve(c["Nq"])
    elif kind in ("forward", "attend"):
        s["plan"] = binding.Forward(c["B"], c["H"], c["Nq"], c["Nk"], c["d"], c["M"], c["C"], c["P"], c["block_q"],
                                    dtype=s["Q"].dtype, flags=binding.FLAG_PARENT_STAYS if c["stays"] else 0)
        if kind == "attend":                                    # the keys were quantised by an earlier call
            s["plan"](s["Q"], s["K"], s["V"], s["Cp"], s["Cc"])
    return s


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "forward":
        return s["plan"](s["Q"], s["K"], s["V"], s["Cp"], s["Cc"])
    if kind == "attend":
        return s["plan"].attend(s["Q"], s["Cp"], s["Cc"])
    if kind == "permuted":
        return binding.forward_permuted(s["Q"], s["K"], s["V"], s["Cp"], s["Cc"], c["P"], c["block_q"], s["perm"])
    if kind == "tiled":
        return binding.forward_tiled(s["Q"], s["K"], s["V"], s["Cp"], s["Cc"], c["P"], c["block_q"], c["tile_m"])
    new = binding.codebook_update(s["K"], s["Cp"], s["Cc"], *s["stats"], 0.99)
    return [*new, *s["stats"]]                                  # the statistics are updated in place


# ------------------------------------------------------------------------------------------------ work
def work(case):
    """Inputs read once, outputs written once, and the products the method is made of (assignment over the
    parents and one parent's children, logits and values over the parents and the refined children)."""
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    BH, d, M, C, P = c["B"] * c["H"], c["d"], c["M"], c["C"], c["P"]
    q, k = BH * c["Nq"], BH * c["Nk"]
    books = c["H"] * M * (1 + C) * d * es
    assign = 2.0 * k * (M + C) * d
    attend = 2.0 * q * (M + P * C) * d * 2
    if c["kind"] == "update":
        stats = 4 * c["H"] * M * (1 + C) * (d + 1)
        return dict(bytes=k * d * es + 2 * books + 2 * stats, flops=assign + k * d)
    if c["kind"] == "attend":
        return dict(bytes=2 * q * d * es + books + BH * M * (1 + C) * (2 * d + 4), flops=attend)
    out = 2 * q * d * es + 2 * k * d * es + books
    if c["kind"] in ("permuted", "tiled"):                      # selection and importance are returned too
        out += BH * math.ceil(c["Nq"] / c["block_q"]) * 4 * (M + P)
    return dict(bytes=out, flops=assign + attend + k * d)


def tolerance(case):
    """About four times the distance of the paths from their 64-bit evaluation (the oracle) on such inputs."""
    if case["kind"] == "update":
        # fp32 sums in another order (1e-6), then one bf16 rounding of the codebooks: a value next to a rounding
        # boundary may move by an ulp (2^-8)
        return dict(rel=2e-4, max=0.02)
    if case["kind"] in ("permuted", "tiled"):
        # measured 1.8e-3 (bf16 weights and values); the returned selection may flip where two parents'
        # importances agree to the last bits of fp32
        return dict(rel=1e-2, differ=2e-3)
    if case["dtype"] == "f32":
        return dict(rel=4e-5)                                   # measured 4e-7 .. 8e-6 (logits up to 100 in the exponent)
    return dict(rel=1e-2)                                       # measured 1.8e-3 .. 2.5e-3
