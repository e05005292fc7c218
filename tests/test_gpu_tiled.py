"""avq_forward_tiled (importance from tiled parents, Eq. "aproxdenom") against the oracle, for codebooks
beyond one tile (M = 512, 1024) and for the degenerate tilings."""
import numpy as np
import pytest
import torch

from oracle import avq_oracle as orc
from paper_2607_12789_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wl,tile_m", [
    (synth.Workload("t512", B=1, H=2, N=1536, d=64, M=512, C=4, P=32, block_q=128, seed=61, alpha=0.3,
                    hot_queries=True), 128),
    (synth.Workload("t1024", B=1, H=1, N=2048, d=64, M=1024, C=4, P=64, block_q=128, seed=62, alpha=0.3,
                    hot_queries=True), 256),
    (synth.Workload("t96", B=2, H=2, N=300, d=32, M=96, C=2, P=9, block_q=50, dtype="f32", seed=63, alpha=0.5), 32),
], ids=["bf16_M512_tile128", "bf16_M1024_tile256", "f32_M96_tile32"])
def test_tiled_selection_importance_and_output_match_the_oracle(wl, tile_m):
    x = synth.generate(wl)
    dv = parity.to_device(x, wl.dtype)
    Y, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q, tile_m,
                                         scale=wl.scale)
    torch.cuda.synchronize()
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, wl.block_q, wl.scale, form="factorised",
                      tile_m=tile_m)
    same, excused = parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)
    assert excused == 0
    rows = np.repeat(same, wl.block_q, axis=-1)[..., :wl.N]
    parity.compare_output(Y.float().cpu().numpy().astype(np.float64), ref["Y"], wl.dtype, rows)
    # the tiling really changed some selections with respect to the exact importance
    exact = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, wl.block_q, wl.scale, form="factorised")
    assert (exact["selected"] != ref["selected"]).any()


def test_one_tile_reproduces_the_plain_forward():
    wl = synth.C0.with_(H=2, seed=64)
    x = synth.generate(wl)
    dv = parity.to_device(x, "f32")
    Y, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q, 32)
    Y0, topp0, imp0, _ = binding.forward(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q, aux=True)
    assert torch.equal(topp, topp0) and torch.allclose(imp, imp0, rtol=1e-5, atol=1e-6)
    assert (Y - Y0).abs().max().item() <= 1e-5


@pytest.mark.parametrize("dtype,d,M,tile_m,N,bq", [("f32", 64, 96, 32, 300, 100), ("f32", 36, 200, 64, 260, 64),
                                                   ("bf16", 64, 256, 128, 300, 128), ("f32", 64, 96, 32, 300, 150)])
def test_a_later_tile_far_above_an_earlier_one_leaves_finite_importances(dtype, d, M, tile_m, N, bq):
    """Logits of the last tile lie about 150 (natural log) above those of the tiles before it, more than fp32's
    exponent holds: the importances of the earlier tiles are ratios of their own and must not come out as 0 / 0."""
    wl = synth.Workload("far_tile", B=1, H=2, N=N, d=d, M=M, C=2, P=max(2, M // 8), block_q=bq, dtype=dtype, seed=65 + M,
                        alpha=0.8)
    x = synth.generate(wl)
    first = (M - 1) // tile_m * tile_m
    u = np.zeros(d, dtype=np.float32)
    u[0] = 1.0
    lift = 150.0 / wl.scale / 32.0
    for k, f in (("Cp", slice(None)), ("Cc", slice(None))):
        x[k][:, first:] += lift * u
    x["K"] += 0.5 * lift * u                                     # half way: keys on both sides
    x["K"][:, :, ::2] += 0.5 * lift * u
    x["K"][:, :, 1::2] -= 0.5 * lift * u
    x["Q"] += 32.0 * u
    x = {k: (synth.round_to_bf16(v) if dtype == "bf16" else v) for k, v in x.items()}
    dv = parity.to_device(x, dtype)
    Y, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, bq, tile_m, scale=wl.scale)
    torch.cuda.synchronize()
    assert torch.isfinite(imp).all()
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, bq, wl.scale, form="factorised", tile_m=tile_m)
    assert (ref["importance"][..., :first] > 0.05).any(axis=-1).all()   # an earlier tile does matter
    same, _ = parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)
    rows = np.repeat(same, bq, axis=-1)[..., :N]
    parity.compare_output(Y.float().cpu().numpy().astype(np.float64), ref["Y"], dtype, rows)


@pytest.mark.parametrize("M,C,P,bq,tile_m,N,flags", [(5, 1, 2, 17, 32, 64, 0),           # one narrow tile, children in one too
                                                     (130, 3, 20, 100, 96, 250, 0),      # ragged tiles of 96, blocks of 100 rows
                                                     (300, 16, 40, 50, 256, 330, 0),     # two code tiles per importance tile
                                                     (256, 2, 32, 64, 64, 300, binding.FLAG_PARENT_STAYS),
                                                     (40, 5, 40, 128, 32, 129, 0),       # every parent refined
                                                     (512, 4, 0, 128, 128, 300, 0)])     # none
def test_tensor_core_tiles_at_their_edges(M, C, P, bq, tile_m, N, flags):
    """bf16, d = 64: importance tiles, code tiles, query blocks and child tiles with remainders."""
    wl = synth.Workload("edges", B=1, H=2, N=N, d=64, M=M, C=C, P=P, block_q=bq, seed=66 + M, alpha=0.5, hot_queries=True)
    x = synth.generate(wl)
    stays = bool(flags & binding.FLAG_PARENT_STAYS)
    if stays:
        x["K"][:, :, ::2] = synth.round_to_bf16((x["Cp"][:, :1] + 0.05 * x["V"][0, :, : len(x["K"][0, 0, ::2])]).astype(np.float32))
    dv = parity.to_device(x, "bf16")
    Y, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, bq, tile_m, scale=wl.scale, flags=flags)
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], P, bq, wl.scale, parent_stays=stays, form="factorised", tile_m=tile_m)
    same, _ = parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)
    rows = np.repeat(same, bq, axis=-1)[..., :N]
    parity.compare_output(Y.float().cpu().numpy().astype(np.float64), ref["Y"], "bf16", rows)


def test_values_that_are_not_finite_leave_the_other_dimensions_alone():
    """A tile with an infinite value sum takes its product on the CUDA cores: an infinity times the part of a weight that
    happens to be zero must not become NaN, and nothing leaks into other dimensions or heads."""
    wl = synth.Workload("inf", B=1, H=2, N=300, d=64, M=256, C=4, P=32, block_q=128, seed=67, alpha=0.5)
    x = synth.generate(wl)
    x["Q"] *= 0.1                                                # every key has some weight
    run = lambda: binding.forward_tiled(*(parity.to_device(x, "bf16")[k] for k in ("Q", "K", "V", "Cp", "Cc")), wl.P, 128, 128,
                                        scale=wl.scale)[0].float().cpu().numpy()
    x["V"][0, 0, 100, 7] = 0.0
    plain = run()
    x["V"][0, 0, 100, 7] = np.inf
    Y = run()
    assert np.isposinf(Y[0, 0, :, 7]).all()
    rest = np.arange(64) != 7
    assert np.array_equal(Y[0, 1], plain[0, 1])
    # the tile's sum in another order (float32), then one bf16 rounding: an ulp (2^-8) where a value is next to a boundary
    assert np.abs(Y[0, 0][:, rest] - plain[0, 0][:, rest]).max() <= 2 ** -8 * np.abs(plain).max()


def _neighbouring_parents_refined(M, C, P, bq, N, seed):
    """Half of the keys close to a parent, half to a child; queries around P parents with consecutive indices, which are then
    the refined ones: with PARENT_STAYS their value rows (the keys that stay) fill whole groups of a tile's columns."""
    wl = synth.Workload("neighbours", B=1, H=2, N=N, d=64, M=M, C=C, P=P, block_q=bq, seed=seed)
    x = synth.generate(wl)
    g = np.random.default_rng(seed)
    for h in range(2):
        hot = M // 4 + np.arange(N) % P
        x["K"][0, h, ::2] = x["Cp"][h, g.permutation(hot)[::2]] + 0.05 * g.standard_normal(((N + 1) // 2, 64))
        x["Q"][0, h] = 0.3 * x["Cp"][h, hot] + 0.3 * g.standard_normal((N, 64))
    return wl, {k: synth.round_to_bf16(v.astype(np.float32)) for k, v in x.items()}


@pytest.mark.parametrize("M,C,P,tile_m", [(512, 8, 64, 128), (512, 16, 48, 256), (160, 16, 100, 32), (1024, 4, 32, 128)])
def test_keys_that_stay_under_refined_neighbours(M, C, P, tile_m):
    """Eight and more code tiles with rows that take 1 + C loads each, in some warps and not in others; forty calls agree."""
    wl, x = _neighbouring_parents_refined(M, C, P, 128, 700, seed=70 + M + C)
    dv = parity.to_device(x, "bf16")
    call = lambda: binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, 128, tile_m, scale=wl.scale,
                                         flags=binding.FLAG_PARENT_STAYS)
    Y, topp, imp = call()
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], P, 128, wl.scale, parent_stays=True, form="factorised", tile_m=tile_m)
    assert (np.diff(ref["selected"][:, :, 0]) == 1).mean() > 0.5 and 100 < (ref["child_idx"] < 0).sum() < 1300
    same, _ = parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)
    rows = np.repeat(same, 128, axis=-1)[..., :wl.N]
    parity.compare_output(Y.float().cpu().numpy().astype(np.float64), ref["Y"], "bf16", rows)
    # (the value sums are added up by atomics, in any order: a last bit of float32, then at most one of bfloat16)
    for _ in range(40):
        Y2, topp2, imp2 = call()
        assert torch.equal(topp, topp2) and torch.equal(imp, imp2)
        assert (Y2.float() - Y.float()).abs().max().item() <= 2 ** -7 * Y.float().abs().max().item()


@pytest.mark.parametrize("M,C,P", [(512, 4, 64), (1024, 8, 64)])
def test_a_value_that_is_not_finite_in_the_first_of_many_tiles(M, C, P):
    """The tile's product then runs on the CUDA cores, slowly, while other warps are up to a turn ahead: six and twelve code tiles,
    so that the descriptions of the tiles are overwritten meanwhile.  The other dimensions are the oracle's."""
    wl = synth.Workload("inf_first", B=1, H=2, N=900, d=64, M=M, C=C, P=P, block_q=128, seed=71 + M, alpha=0.8)
    x = synth.generate(wl)
    x["Q"] = synth.round_to_bf16(0.1 * x["Q"])                   # every key has some weight
    dv = parity.to_device(x, "bf16")
    first = int((binding.assign(dv["K"], dv["Cp"], dv["Cc"], flags=binding.FLAG_SIMT)[0][0, 0] < 128).nonzero()[0])
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], P, 128, wl.scale, form="factorised", tile_m=128)
    dv["V"][0, 0, first, 7] = float("inf")
    Y, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, 128, 128, scale=wl.scale)
    same, _ = parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)
    rows = np.repeat(same, 128, axis=-1)[..., :wl.N]
    Y = Y.float().cpu().numpy().astype(np.float64)
    assert np.isposinf(Y[0, 0, :, 7]).all()
    Y[0, 0, :, 7] = ref["Y"][0, 0, :, 7]
    parity.compare_output(Y, ref["Y"], "bf16", rows)


@pytest.mark.parametrize("M,C,P,tile_m", [(1024, 8, 128, 256), (96, 16, 96, 96)])
def test_many_tiles_in_many_blocks_come_out_the_same_every_time(M, C, P, tile_m):
    """Sixteen and thirteen code tiles in 96 blocks, each tile's logits above those of the tile before it in half of the rows:
    were a warp to take a maximum of another turn, its weights would be off by powers of e."""
    wl = synth.Workload("ladder", B=2, H=3, N=2048, d=64, M=M, C=C, P=P, block_q=128, seed=72 + M, alpha=0.8)
    x = synth.generate(wl)
    lift = np.zeros((M, 64), dtype=np.float32)
    lift[:, 0] = 8.0 * np.arange(M) / M
    x["Cp"], x["Cc"] = x["Cp"] + lift, x["Cc"] + lift[:, None]
    x["Q"][..., ::2, 0] += 6.0
    x["Q"][..., 1::2, 0] -= 6.0
    x = {k: synth.round_to_bf16(v) for k, v in x.items()}
    dv = parity.to_device(x, "bf16")
    call = lambda: binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, 128, tile_m, scale=wl.scale)
    Y, topp, imp = call()
    for _ in range(40):
        Y2, topp2, imp2 = call()
        assert torch.equal(topp, topp2) and torch.equal(imp, imp2)
        assert (Y2.float() - Y.float()).abs().max().item() <= 2 ** -7 * Y.float().abs().max().item()
    ref = orc.forward_head(x["Q"][1, 2], x["K"][1, 2], x["V"][1, 2], x["Cp"][2], x["Cc"][2], P, 128, wl.scale, form="factorised",
                           tile_m=tile_m)
    head = lambda t: t.float().cpu().numpy()[1, 2]
    same, _ = parity.compare_selection(dict(selected=topp.cpu().numpy()[1, 2], importance=head(imp)), ref)
    parity.compare_output(head(Y).astype(np.float64), ref["Y"], "bf16", np.repeat(same, 128))


@pytest.mark.parametrize("bq,P,bad", [(64, 32, float("nan")), (100, 32, float("inf")), (50, 0, float("nan"))])
def test_a_query_that_is_not_finite_spoils_no_other_block(bq, P, bad):
    """Blocks of fewer than 128 queries: the tile's further rows hold the next block's queries, which must not count here."""
    wl = synth.Workload("bad_query", B=1, H=2, N=400, d=64, M=256, C=4, P=P, block_q=bq, seed=73 + bq, alpha=0.5)
    x = synth.generate(wl)
    run = lambda q: binding.forward_tiled(q, *(dv[k] for k in ("K", "V", "Cp", "Cc")), P, bq, 128, scale=wl.scale)
    dv = parity.to_device(x, "bf16")
    Y0, topp0, imp0 = run(dv["Q"])
    Q = dv["Q"].clone()
    Q[0, 0, bq + 3] = bad                                        # in block 1 of head 0 only
    Y, topp, imp = run(Q)
    assert not torch.isfinite(Y[0, 0, bq + 3]).any()
    keep = torch.ones(1, 2, imp.shape[2], dtype=torch.bool, device="cuda")
    keep[0, 0, 1] = False
    assert torch.equal(imp[keep], imp0[keep]) and torch.equal(topp[keep], topp0[keep])
    rows = keep.repeat_interleave(bq, dim=-1)[..., :400]
    # (value sums added up in any order: at most an ulp of bfloat16)
    assert (Y.float() - Y0.float())[rows].abs().max().item() <= 2 ** -7 * Y0.float().abs().max().item()


@pytest.mark.parametrize("M,C,P,bq,tile_m,flags", [(768, 8, 64, 128, 128, 0), (544, 3, 50, 100, 160, 0),
                                                   (768, 8, 64, 128, 256, binding.FLAG_PARENT_STAYS)])
def test_the_cuda_core_flag_selects_the_cuda_core_kernel_and_both_agree(M, C, P, bq, tile_m, flags):
    wl = synth.Workload("both", B=1, H=2, N=1000, d=64, M=M, C=C, P=P, block_q=bq, seed=74 + M, alpha=0.8, hot_queries=True)
    dv = parity.to_device(synth.generate(wl), "bf16")
    call = lambda f: binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, bq, tile_m, scale=wl.scale, flags=flags | f)
    Y, topp, imp = call(0)
    Y1, topp1, imp1 = call(binding.FLAG_SIMT)
    # importances added up in another order: float32's last bits differ somewhere, and no more than those of some thousand terms
    assert not torch.equal(imp, imp1) and torch.allclose(imp, imp1, rtol=2e-4, atol=1e-5)
    same = (topp == topp1).all(-1)
    assert same.float().mean().item() > 0.9                      # (a near-tie may fall either way)
    rows = same.repeat_interleave(bq, dim=-1)[..., :wl.N]
    # one bfloat16 rounding each: an ulp where float32 results fall on either side of a boundary
    assert ((Y.float() - Y1.float()).abs()[rows] <= 2 ** -7 * Y1.float().abs()[rows] + 1e-5).all()


@pytest.mark.parametrize("M,C,P,bq,tile_m,tensor", [(64, 4, 8, 128, 64, False), (64, 4, 8, 128, 32, True), (64, 4, 16, 65, 64, True),
                                                    (63, 4, 16, 128, 256, False), (65, 1, 0, 128, 128, True), (32, 3, 20, 100, 32, False),
                                                    (33, 1, 2, 100, 32, True), (160, 4, 19, 64, 128, False), (160, 4, 20, 64, 128, True),
                                                    (64, 4, 8, 16, 32, False), (512, 4, 64, 16, 128, True)])
def test_small_codebooks_and_blocks_stay_on_the_cuda_cores(M, C, P, bq, tile_m, tensor):
    """Where the tensor-core kernel takes longer (up to 1.5 times at 64 parents and blocks of 8 to 64 queries) it is not used: the
    importances then are those of the CUDA-core kernel bit for bit; elsewhere some last bit differs."""
    wl = synth.Workload("rule", B=1, H=4, N=500, d=64, M=M, C=C, P=P, block_q=bq, seed=75 + M, alpha=0.8, hot_queries=True)
    dv = parity.to_device(synth.generate(wl), "bf16")
    call = lambda f: binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, bq, tile_m, scale=wl.scale, flags=f)
    (Y, _, imp), (Y1, _, imp1) = call(0), call(binding.FLAG_SIMT)
    assert torch.equal(imp, imp1) == (not tensor)
    assert torch.allclose(imp, imp1, rtol=2e-4, atol=1e-5)
    assert ((Y.float() - Y1.float()).abs() <= 2 ** -7 * Y1.float().abs() + 1e-5).float().mean().item() > 0.98   # (near-tied selections)


def test_the_value_product_rounds_like_float32_multiply_adds():
    """Three parents with the same weight w and value sums a, b and -(a + b) of 24 significant bits: the output is what the value
    product rounds off.  Three float32 multiply-adds leave 0.36 2^-24 w (root mean square, on these numbers), products of
    bfloat16 parts 0.46 where the parts are cut off and 0.10 where they are rounded to nearest."""
    g = np.random.default_rng(76)
    M, N, d = 128, 128, 64
    rng = lambda n: g.integers(2 ** 23, 2 ** 24, n)
    a = rng(d) * 2.0 ** -25                                      # in [1/4, 1/2), multiples of 2^-25
    b = (rng(d) // 2 * 2 * 2.0 ** -25) + (a * 2.0 ** 25 % 2) * 2.0 ** -25   # a + b: a multiple of 2^-24
    x = np.stack([np.zeros(d), a, b, -(a + b)])
    assert (x.astype(np.float32) == x).all()
    parts, rest = [], x.copy()                                   # each as the sum of three bfloat16: the values of three keys
    for _ in range(3):
        p = synth.round_to_bf16(rest.astype(np.float32)).astype(np.float64)
        parts.append(p)
        rest = rest - p
    assert (rest == 0).all()
    Cp = np.zeros((M, d))
    Cp[:, 1] = np.arange(M) * 4.0 + 100.0                        # far away and without keys
    for j in range(4):
        Cp[j] = 0.0
        Cp[j, 2 + j] = 8.0                                       # (queries are zero there)
    Cp[0, 0] = 2.0
    Cp[1:4, 0] = 1.0
    K = np.repeat(Cp[:4], 3, axis=0)
    V = np.stack([parts[i][j] for j in range(4) for i in range(3)])
    Q = np.zeros((N, d))
    Q[:, 0] = 8.0 * (0.05 + 3.0 * g.random(N))
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v[None])).float().cuda().to(torch.bfloat16)
    Q, K, V, Cp_ = t(Q[None]), t(K[None]), t(V[None]), t(Cp)
    Y, _, _ = binding.forward_tiled(Q, K, V, Cp_, Cp_[:, :, None].contiguous(), 0, 128, 128, scale=0.125)
    w = np.exp(-Q[0, 0, :, 0].double().cpu().numpy() / 8)
    left = Y[0, 0].double().cpu().numpy() * ((3 + 9 * w) / w)[:, None]      # times the denominator, over the weight
    rms = np.sqrt((left ** 2).mean()) * 2.0 ** 24
    print(f"rms {rms:.2f} 2^-24")
    assert 0 < rms <= 0.36


def test_value_sums_beyond_the_largest_bfloat16():
    """A finite float32 sum that rounds to infinity as a bfloat16 is not split: the output stays finite."""
    wl = synth.Workload("large", B=1, H=1, N=256, d=64, M=256, C=4, P=0, block_q=128, seed=77, alpha=0.5)
    x = synth.generate(wl)
    x["Q"] = synth.round_to_bf16(0.1 * x["Q"])
    dv = parity.to_device(x, "bf16")
    par = binding.assign(dv["K"], dv["Cp"], dv["Cc"], flags=binding.FLAG_SIMT)[0][0, 0]
    two = (par == par[0]).nonzero().flatten()[:2].tolist()
    assert len(two) == 2
    dv["V"][0, 0, :, 7] = 0.0
    dv["V"][0, 0, two[0], 7], dv["V"][0, 0, two[1], 7] = 3.3895e38, 1.2e36   # the largest bfloat16, and less than half a step
    call = lambda f: binding.forward_tiled(*(dv[k] for k in ("Q", "K", "V", "Cp", "Cc")), 0, 128, 128, scale=wl.scale, flags=f)[0]
    Y, Y1 = call(0).float(), call(binding.FLAG_SIMT).float()
    assert torch.isfinite(Y).all() and (Y[..., 7] > 1e34).all()
    # one bfloat16 rounding each
    assert ((Y - Y1).abs() <= 2 ** -7 * Y1.abs() + 1e-5).all()
