"""GPU parity of the tcgen05 tensor-core path (bf16) against the fp64 oracle.

Small and mid-size configurations are compared whole; the long ones on whole sampled heads
(assignments, aggregates) and sampled query blocks (importance, top-P, output)."""
import numpy as np
import pytest
import torch

from paper_2607_12789_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu


def test_small_bf16_single_child_tile():
    rep = parity.full_parity(synth.C1.with_(B=1, H=2, N=512))
    assert rep["empty_parents"] > 0


def test_c1_vitb_full():
    rep = parity.full_parity(synth.C1)
    print("c1", rep)


def test_c2_mid_full():
    rep = parity.full_parity(synth.C2)
    print("c2", rep)


def test_c3_long_sampled():
    rep, gpu, x = parity.sampled_parity(synth.C3, heads=[(0, 3), (0, 12)], blocks_per_head=8)
    print("c3", rep)
    # properties that hold at any size, over the whole tensor
    assert np.isfinite(gpu["Y"]).all()
    assert np.array_equal(gpu["np"].sum(axis=-1), np.full((1, 16), 16384.0))
    assert np.array_equal(gpu["nc"].sum(axis=-1), gpu["np"])
    np.testing.assert_allclose(gpu["importance"].sum(axis=-1), 128.0, rtol=1e-4)
    np.testing.assert_allclose(gpu["Vp"].sum(axis=2), x["V"].astype(np.float64).sum(axis=2), atol=5e-3)
    # every query tile of six heads against the factorised oracle (768 of the 2048 tiles)
    rep2, _ = parity.heads_parity_factorised(synth.C3, [(0, h) for h in (0, 3, 6, 9, 12, 15)], x=x, gpu=gpu)
    print("c3 whole heads", rep2)
    assert rep2["blocks"] >= 6 * 128 - rep2["topp_flips_excused"]


# Sweep configuration: every (N, M, P) point has a parity test.  All P of one (N, M) share their data, so
# the oracle's assignment of a head is computed once per (N, M).  N <= 16384: every query tile of the
# listed heads (factorised oracle); N = 65536: one head, every tile.
@pytest.mark.parametrize("M", [32, 64, 128, 256])
def test_sweep_N1024_all_P(M):
    for P in synth.sweep_P(M):
        parity.full_parity(synth.sweep_point(1024, M, P).with_(H=4))


@pytest.mark.parametrize("M", [32, 64, 128, 256])
@pytest.mark.parametrize("N,H", [(4096, 2), (16384, 1), (65536, 1)])
def test_sweep_all_P_whole_heads(N, H, M):
    wl0 = synth.sweep_point(N, M, 0).with_(H=H)
    x = synth.generate(wl0)
    heads = [(0, h) for h in range(H)]
    cache = {}
    for P in synth.sweep_P(M):
        rep, cache = parity.heads_parity_factorised(wl0.with_(P=P), heads, x=x, assignments=cache, P=P)
        print(f"sweep N={N} M={M} P={P}", rep)


def test_sweep_dense_definition_on_sampled_tiles():
    """The O(N^2) definition itself on sampled tiles of long sweep points."""
    parity.sampled_parity(synth.sweep_point(16384, 256, 32), heads=[(0, 5)], blocks_per_head=6)
    parity.sampled_parity(synth.sweep_point(65536, 64, 16), heads=[(0, 9)], blocks_per_head=4)


def _exact_grid(g, shape, step=0.25, lim=4.0):
    """Random values on a coarse grid: exactly representable in bf16, sums of squares exact in fp32."""
    return (np.clip(np.round(g.normal(size=shape) / step), -lim / step, lim / step) * step).astype(np.float32)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("C", [4, 8])
def test_exact_ties_on_the_tensor_core_path(d, C):
    """Duplicated parent codewords, duplicated children, keys at exact midpoints and keys equal to
    codewords, inside the tcgen05 envelope (M = 32): best and runner-up distances coincide, so the
    float64 recheck of avq_assign decides, and the lowest index must win (Algorithm 1's strict '<')."""
    from oracle import avq_oracle as orc
    g = np.random.default_rng(7 + d + C)
    M = 32
    base = _exact_grid(g, (12, d))
    Cp = base[g.integers(0, 12, size=M)]                      # 32 parents drawn from 12 distinct rows
    Cp[5] = Cp[2]; Cp[9] = Cp[2]; Cp[31] = Cp[30]
    Cc = np.repeat(Cp[:, None, :], C, axis=1).copy()
    Cc[:, C // 2:] += 0.5                                     # children 0..C/2-1 equal, C/2..C-1 equal
    Cc[3] = _exact_grid(g, (C, d))
    Cc[3, 2] = Cc[3, 1]                                       # a duplicated pair in the middle
    keys = [Cp,                                               # keys on parent codewords
            Cc.reshape(-1, d),                                # keys on child codewords
            0.5 * (Cp[:16] + Cp[16:]),                        # exact midpoints of two parents
            0.5 * (Cc[:, 0] + Cc[:, C - 1]),                  # exact midpoints of two children
            _exact_grid(g, (200, d))]
    K = np.concatenate(keys).astype(np.float32)
    assert np.array_equal(synth.round_to_bf16(K), K) and np.array_equal(synth.round_to_bf16(Cc), Cc)
    ref = orc.assign_head(K, Cp, Cc)
    assert (ref["parent_margin"] == 0).sum() >= M and (ref["child_margin"] == 0).sum() >= M
    # a key that sits on parent i must be given the FIRST parent with that codeword (written out by hand)
    first_equal = [min(j for j in range(M) if np.array_equal(Cp[j], Cp[i])) for i in range(M)]
    assert ref["parent_idx"][:M].tolist() == first_equal and first_equal[5] == first_equal[9] == first_equal[2]
    assert len(set(first_equal)) <= 12
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(torch.bfloat16)
    pi, ci = binding.assign(t(K[None, None]), t(Cp[None]), t(Cc[None]))
    torch.cuda.synchronize()
    assert np.array_equal(pi.cpu().numpy()[0, 0], ref["parent_idx"])
    assert np.array_equal(ci.cpu().numpy()[0, 0], ref["child_idx"])


def test_ragged_tail_and_nq_not_nk():
    wl = synth.C1.with_(B=1, H=3, N=1000, seed=31)
    x = synth.generate(wl)
    x["Q"] = np.ascontiguousarray(x["Q"][:, :, :700])
    parity.full_parity(wl, x=x)


def test_other_shapes_d128_C8_M96():
    parity.full_parity(synth.Workload("odd", B=1, H=2, N=768, d=128, M=96, C=8, P=12, block_q=128, seed=77,
                                      alpha=0.5, hot_queries=True))


@pytest.mark.parametrize("wl", [synth.C1.with_(B=2, H=2, N=1500, seed=51), synth.C3.with_(H=2, N=2000, seed=52),
                                synth.C2.with_(B=1, H=2, N=1100, seed=53),
                                synth.sweep_point(4096, 32, 8).with_(H=2, seed=54),      # long head: leaf-ordered aggregate
                                synth.sweep_point(4096, 128, 128).with_(H=2, seed=55)],  # every parent refined, 4 child chunks
                         ids=["d64_M64_C4", "d128_M256_C4", "d64_M128_C8", "long_head_M32", "all_refined_M128"])
def test_parent_stays_on_the_tensor_core_path(wl):
    """Algorithm 1's masked scatter on the tcgen05 path: half of the keys hug their parent and stay with it
    (child index -1), the others move to a child; a refined parent keeps the stay residual."""
    x = synth.generate(wl)
    g = np.random.default_rng(wl.seed)
    for b in range(wl.B):
        for h in range(wl.H):
            near = x["Cp"][h][g.integers(0, wl.M, wl.N // 2)] + 0.05 * g.standard_normal((wl.N // 2, wl.d))
            x["K"][b, h, ::2] = synth.round_to_bf16(near.astype(np.float32))[: len(x["K"][b, h, ::2])]
    rep = parity.full_parity(wl, flags=binding.FLAG_PARENT_STAYS, parent_stays=True, x=x)
    print("stays", rep)
    total = wl.B * wl.H * wl.N
    assert 0.3 * total <= rep["stay_count"] <= 0.7 * total        # a real mixture of stayed and moved keys
    # and the two rules really differ on this input
    gpu_rep = parity.gpu_forward(wl, x, flags=0)
    gpu_st = parity.gpu_forward(wl, x, flags=binding.FLAG_PARENT_STAYS)
    assert (gpu_rep["child_idx"] >= 0).all() and (gpu_st["child_idx"] < 0).any()
    assert np.abs(gpu_rep["Y"] - gpu_st["Y"]).max() > 1e-3


@pytest.mark.parametrize("d,M,C", [(64, 32, 8), (64, 256, 4), (128, 96, 4), (128, 128, 8)])
@pytest.mark.parametrize("spread", ["one_parent", "all_parents", "two_per_sixteen"])
def test_parent_stays_with_few_and_many_parents_per_tile(d, M, C, spread):
    """The child step takes a tile's keys in the order of their parents, 16 per warp: a tile of one parent, tiles whose keys
    have a parent each, and a ragged last tile, half of the keys close to their parent."""
    from oracle import avq_oracle as orc
    g = np.random.default_rng(d + M + C)
    N = 333
    Cp = synth.round_to_bf16(3 * g.standard_normal((M, d)).astype(np.float32))
    Cc = synth.round_to_bf16((Cp[:, None] + 0.8 * g.standard_normal((M, C, d))).astype(np.float32))
    par = {"one_parent": np.full(N, M - 1), "all_parents": g.permutation(N) % M, "two_per_sixteen": np.arange(N) // 8 % M}[spread]
    K = Cc[par, g.integers(0, C, N)] + 0.2 * g.standard_normal((N, d))
    K[::2] = Cp[par[::2]] + 0.05 * g.standard_normal((len(K[::2]), d))
    K = synth.round_to_bf16(K.astype(np.float32))
    ref = orc.assign_head(K, Cp, Cc, parent_stays=True)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a[None])).cuda().to(torch.bfloat16)
    pi, ci = binding.assign(t(K[None]), t(Cp), t(Cc), flags=binding.FLAG_PARENT_STAYS)
    assert np.array_equal(pi.cpu().numpy()[0, 0], ref["parent_idx"])
    assert np.array_equal(ci.cpu().numpy()[0, 0], ref["child_idx"])


def test_tensor_core_and_cuda_core_paths_agree_at_full_size():
    wl = synth.C3.with_(H=4)
    dv = parity.to_device(synth.generate(wl), "bf16")
    args = (dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q)
    Yt, St, Wt, It = binding.forward(*args, scale=wl.scale, aux=True)
    Ys, Ss, Ws, Is = binding.forward(*args, scale=wl.scale, flags=binding.FLAG_SIMT, aux=True)
    assert torch.equal(It["parent_idx"], Is["parent_idx"]) and torch.equal(It["child_idx"], Is["child_idx"])
    assert torch.equal(It["np"], Is["np"]) and torch.equal(It["nc"], Is["nc"])
    same = (St == Ss).all(dim=-1)
    assert same.float().mean() > 0.99                      # selections may differ only at near-ties
    rows = same.repeat_interleave(wl.block_q, dim=-1)
    diff = (Yt.float() - Ys.float()).abs()[rows]
    assert diff.max() <= 2e-2


@pytest.mark.parametrize("H,N,d,M,C", [(2, 40001, 64, 32, 4), (2, 80003, 128, 32, 8), (16, 16384, 64, 64, 4),
                                       (1, 1300000, 64, 256, 8)])
def test_aggregate_long_heads_few_leaves(H, N, d, M, C):
    """avq_aggregate where every leaf collects many keys (the chunked, leaf-ordered variant), ragged
    lengths, skewed and empty leaves: counts exact, sums within fp32 accumulation error of the oracle."""
    from oracle import avq_oracle as orc
    g = np.random.default_rng(100 + N)
    V = synth.round_to_bf16(g.standard_normal((1, H, N, d)).astype(np.float32))
    # skewed leaves: a few popular ones, some never used
    pm = g.dirichlet(np.full(M, 0.3))
    pidx = g.choice(M, size=(1, H, N), p=pm).astype(np.int32)
    cidx = np.minimum(g.geometric(0.5, size=(1, H, N)) - 1, C - 1).astype(np.int32)
    dev = dict(V=torch.from_numpy(V).cuda().to(torch.bfloat16), p=torch.from_numpy(pidx).cuda(),
               c=torch.from_numpy(cidx).cuda())
    Vp, n_p, Vc, n_c = binding.aggregate(dev["V"], dev["p"], dev["c"], M, C)
    torch.cuda.synchronize()
    for h in range(H):
        rVp, rnp, rVc, rnc = orc.aggregate_head(V[0, h], pidx[0, h], cidx[0, h], M, C)
        assert np.array_equal(n_p[0, h].cpu().numpy(), rnp)
        assert np.array_equal(n_c[0, h].cpu().numpy(), rnc)
        scale = 1e-6 * np.sqrt(np.maximum(rnc, 1.0))[..., None] * 50 + 1e-5 * np.abs(rVc)
        assert (np.abs(Vc[0, h].cpu().numpy() - rVc) <= scale + 1e-4).all()
        assert np.allclose(Vp[0, h].cpu().numpy(), rVp, rtol=2e-5, atol=2e-3)


def _random_shapes(n, seed):
    g = np.random.default_rng(seed)
    out = []
    for i in range(n):
        d = int(g.choice([64, 128]))
        C = int(g.choice([4, 8]))
        M = int(g.choice([32, 64, 96, 128, 160, 256]))
        P = int(g.choice([0, 1, M // 8, M // 4, M]))
        H = int(g.integers(1, 4))
        B = int(g.integers(1, 3))
        N = int(g.integers(129, 1400))
        out.append(synth.Workload(f"rnd{i}", B=B, H=H, N=N, d=d, M=M, C=C, P=P, block_q=128, seed=500 + i,
                                  alpha=float(g.choice([0.3, 0.8])), hot_queries=bool(g.integers(0, 2))))
    return out


@pytest.mark.parametrize("wl", _random_shapes(12, seed=20261), ids=lambda w: f"{w.name}-B{w.B}H{w.H}N{w.N}d{w.d}M{w.M}C{w.C}P{w.P}")
def test_random_shapes_full_parity(wl):
    """Seeded random shapes inside the tensor-core envelope (ragged lengths, every d, C, several M and P,
    endpoints included): every stage against the oracle, whole tensors."""
    parity.full_parity(wl)


@pytest.mark.parametrize("C,P", [(4, 4), (4, 17), (8, 32)])
@pytest.mark.parametrize("flags", [0, binding.FLAG_PARENT_STAYS])
def test_smallest_codebook_over_chained_tiles(C, P, flags):
    """32 parents with more tiles than small grids have: one child chunk of 16 columns, several chunks with a ragged last
    one, every parent refined; more tiles than CTAs, and children that move the reference."""
    wl = synth.Workload("m32", B=3, H=16, N=1700, d=64, M=32, C=C, P=P, block_q=128, seed=58 + C + P, alpha=0.6,
                        hot_queries=True, sigma_c=0.5 if P < 32 else 20.0)
    x = synth.generate(wl)
    if flags:                                                     # every other key hugs a parent: it stays
        x["K"][:, :, ::2] = synth.round_to_bf16(x["Cp"][np.arange(16)[None, :, None], np.arange(0, 1700, 2)[None, None] % 32]
                                                + np.float32(0.03))
    parity.full_parity(wl, flags=flags, parent_stays=bool(flags), x=x)


def test_long_ragged_head_uses_chunked_aggregate_end_to_end():
    """A ragged long head over few leaves (the chunked aggregate inside avq_forward), sampled against the oracle."""
    wl = synth.sweep_point(16384, 32, 4).with_(H=2, N=16384 + 77, name="ragged_long")
    parity.sampled_parity(wl, heads=[(0, 1)], blocks_per_head=4)


def test_degenerate_all_keys_on_one_codeword():
    """Every key equals one parent codeword: that parent holds all keys, every other parent is empty, the
    importances are zero but one, and the top-P set is that parent plus the lowest-index empty ones (the
    tie rule across a whole group of equal importances); empty children must not disturb the maxima."""
    wl = synth.C1.with_(B=1, H=2, N=512, seed=41)
    x = synth.generate(wl)
    for h in range(wl.H):
        x["K"][0, h, :, :] = x["Cp"][h, 5]
    rep = parity.full_parity(wl, x=x)
    assert rep["empty_parents"] == wl.H * (wl.M - 1)
    assert rep["topp_flips_excused"] == 0


def test_single_query_block_shorter_than_a_tile_and_tiny_key_set():
    """Nq = 1 and Nk = 5: one ragged query tile, one ragged key tile, almost every codeword empty."""
    wl = synth.C1.with_(B=1, H=1, N=5, seed=43)
    x = synth.generate(wl)
    x["Q"] = np.ascontiguousarray(x["Q"][:, :, :1])
    parity.full_parity(wl, x=x)


def test_chained_tiles_with_several_child_chunks():
    """More tiles than one wave of CTAs (every CTA takes several tiles in a row) with every parent refined, so
    that each tile runs through several child chunks before the next tile's loads are issued."""
    parity.sampled_parity(synth.sweep_point(16384, 64, 64), heads=[(0, 7)], blocks_per_head=4)
    parity.sampled_parity(synth.sweep_point(16384, 256, 64).with_(H=4), heads=[(0, 2)], blocks_per_head=3)


@pytest.mark.parametrize("d,M,C,P,N", [(64, 64, 4, 16, 300), (64, 96, 8, 40, 260), (128, 64, 4, 5, 250), (128, 256, 4, 48, 400),
                                       (64, 160, 4, 33, 257)])
def test_children_far_above_the_parents_move_the_reference(d, M, C, P, N):
    """Children so far from their parents that their logits exceed the parents' maximum by more than 64 powers of two:
    the attention kernel's rescaling turn, in every tile plan, over one and several child chunks.  (P small against a tile of few queries
    is left out: the P-th importance then lies below 2^-126, the smallest weight fp32 holds, and the choice is open.)"""
    wl = synth.Workload("far", B=1, H=2, N=N, d=d, M=M, C=C, P=P, block_q=128, seed=900 + M + d, alpha=0.6,
                        hot_queries=True, sigma_c=20.0)
    x = synth.generate(wl)
    s = np.einsum("hnd,hmd->hnm", x["Q"][0].astype(np.float64), x["Cp"].astype(np.float64)).max(-1)
    c = np.einsum("hnd,hmcd->hnmc", x["Q"][0].astype(np.float64), x["Cc"].astype(np.float64)).max((-1, -2))
    assert ((c - s) * wl.scale * np.log2(np.e) > 80).mean() > 0.5
    parity.full_parity(wl, x=x)


@pytest.mark.parametrize("d,M,C,P,N", [(64, 64, 4, 16, 300), (64, 96, 8, 40, 260), (128, 64, 4, 5, 250), (128, 256, 4, 48, 400),
                                       (64, 160, 4, 33, 300)])
def test_large_values_leave_room_for_children_above_their_parents(d, M, C, P, N):
    """Values of 1e28 under children whose logits exceed the parents' maximum by tens of powers of two: the running sums
    must move to the children's reference before they leave fp32's range.  (The output is compared divided by 1e28, which
    bf16 inputs and fp32 sums carry without a rounding of their own; avq_attend over the same workspace agrees.)"""
    wl = synth.Workload("large", B=1, H=2, N=N, d=d, M=M, C=C, P=P, block_q=128, seed=950 + M + d, alpha=0.6,
                        hot_queries=True, sigma_c=7.0)
    x = synth.generate(wl)
    s = np.einsum("hnd,hmd->hnm", x["Q"][0].astype(np.float64), x["Cp"].astype(np.float64)).max(-1)
    c = np.einsum("hnd,hmcd->hnmc", x["Q"][0].astype(np.float64), x["Cc"].astype(np.float64)).max((-1, -2))
    gap = (c - s) * wl.scale * np.log2(np.e)
    assert ((gap > 40) & (gap < 62)).mean() > 0.2
    unit = float(2.0 ** 93)                                      # 9.9e27
    dv = parity.to_device(x, "bf16")
    dv["V"] = (dv["V"].float() * unit).to(torch.bfloat16)
    f = binding.Forward(1, 2, N, N, d, M, C, P, 128, scale=wl.scale, aux=True)
    Y = f(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"])
    f.check()
    Y2 = f.attend(dv["Q"], dv["Cp"], dv["Cc"])
    assert torch.equal(Y2, Y)
    from oracle import avq_oracle as orc
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], P, 128, wl.scale, form="factorised")
    same, _ = parity.compare_selection(dict(selected=f.topp.cpu().numpy(), importance=f.importance.cpu().numpy()), ref)
    parity.compare_output((Y.double() / unit).cpu().numpy(), ref["Y"], "bf16", np.repeat(same, 128, axis=-1)[..., :N])


@pytest.mark.parametrize("B,d,M,C", [(1, 64, 32, 4), (1, 64, 128, 8), (1, 128, 256, 4), (300, 64, 32, 4), (160, 128, 64, 4)])
def test_a_refined_parent_with_an_infinite_mean_takes_no_part(B, d, M, C):
    """Every parent refined.  The sums of half of the parents leave fp32's range although their children's do not, and no
    query looks that way: the parents' mean rows are infinite, carry no weight and must not reach the output (alone and
    over chained tiles of one CTA)."""
    g = np.random.default_rng(d + M)
    N, H = M * C, 1
    Cp = (3.0 * g.standard_normal((H, M, d))).astype(np.float32)
    Cp[:, : M // 2, 0], Cp[:, M // 2:, 0] = 40.0, -40.0
    Cc = Cp[:, :, None, :] + g.standard_normal((H, M, C, d)).astype(np.float32)
    Cc[..., 0] = Cp[:, :, None, 0]
    K = Cc.reshape(1, H, N, d).repeat(B, 0)                      # one key on every child
    V = g.standard_normal((B, H, N, d)).astype(np.float32)
    V[:, :, N // 2:] = 3e38
    Q = g.standard_normal((B, H, 200, d)).astype(np.float32)
    Q[..., 0] = 40.0                                             # logits of the second half lie 280 (natural log) or more below
    x = {k: synth.round_to_bf16(np.ascontiguousarray(v)) for k, v in dict(Q=Q, K=K, V=V, Cp=Cp, Cc=Cc).items()}
    x["V"] = np.minimum(x["V"], np.float32(3.3e38))
    dv = parity.to_device(x, "bf16")
    Y, topp, imp, inter = binding.forward(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], M, 128, aux=True)
    assert not torch.isfinite(inter["Vp"]).all() and torch.isfinite(inter["Vc"]).all()
    from oracle import avq_oracle as orc
    for b in sorted({0, B - 1}):
        ref = orc.forward(x["Q"][b:b + 1], x["K"][b:b + 1], x["V"][b:b + 1], x["Cp"], x["Cc"], M, 128, 1 / np.sqrt(d),
                          form="factorised")
        parity.compare_output(Y[b:b + 1].double().cpu().numpy(), ref["Y"], "bf16")
    assert torch.isfinite(Y.float()).all()


def test_an_infinite_value_stays_in_its_dimension():
    """One key's value is infinite in one dimension; its parent is refined.  Every query gives its child some weight: that
    dimension of the output is infinite, the others are what they are without it."""
    wl = synth.C1.with_(B=1, H=2, N=512, seed=57, P=64)
    x = synth.generate(wl)
    x["Q"] *= 0.1
    x["V"][0, :, 100, 7] = 0.0
    ref = parity.gpu_forward(wl, x)["Y"]
    x["V"][0, :, 100, 7] = np.inf
    Y = parity.gpu_forward(wl, x)["Y"]
    assert np.isposinf(Y[..., 7]).all()
    rest = np.arange(64) != 7
    assert np.abs(Y[..., rest] - ref[..., rest]).max() <= 1.6e-2   # (a mean next to a rounding boundary: an ulp of bf16)


@pytest.mark.parametrize("M,C,P", [(32, 4, 4), (32, 8, 9), (64, 4, 8), (96, 8, 12), (128, 4, 16)])
def test_selection_of_a_head_does_not_depend_on_the_rest_of_the_call(M, C, P):
    """One image alone (a grid that leaves the chip idle takes twice the warps per tile) and the same image in a batch:
    the importances agree to the last bit, and so do the selections."""
    wl = synth.Workload("alone", B=5, H=12, N=785, d=64, M=M, C=C, P=P, block_q=128, seed=77 + M, alpha=0.5)
    dv = parity.to_device(synth.generate(wl), "bf16")
    _, topp, imp, _ = binding.forward(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, 128, aux=True)
    for b in (0, 3):
        one = {k: dv[k][b:b + 1].contiguous() for k in "QKV"}
        _, topp1, imp1, _ = binding.forward(one["Q"], one["K"], one["V"], dv["Cp"], dv["Cc"], P, 128, aux=True)
        assert torch.equal(imp1[0], imp[b]) and torch.equal(topp1[0], topp[b])


def _offset_inputs(B, H, N, d, M, C, offset, seed, twice=True):
    """Half of the keys hug their parent, half a child; some children stand there twice; everything shifted by `offset`."""
    g = np.random.default_rng(seed)
    Cp = 3 * g.standard_normal((H, M, d))
    Cc = Cp[:, :, None] + 1.2 * g.standard_normal((H, M, C, d))
    if twice:
        Cc[:, ::3, C - 1] = Cc[:, ::3, 0]
    par, chi = g.integers(0, M, (B, H, N)), g.integers(0, C, (B, H, N))
    head = np.arange(H)[None, :, None]
    K = np.where((np.arange(N) % 2 == 0)[:, None], Cp[head, par], Cc[head, par, chi]) + 0.05 * g.standard_normal((B, H, N, d))
    dev = lambda a: (torch.from_numpy(a).float().cuda() + offset).to(torch.bfloat16)
    return dev(K), dev(Cp), dev(Cc)


@pytest.mark.parametrize("B,H,N,d,M,C", [(1, 16, 4736, 64, 64, 4), (2, 16, 2400, 64, 96, 8), (1, 16, 4736, 128, 64, 8),
                                         (1, 16, 9500, 128, 256, 4)])
@pytest.mark.parametrize("flags", [0, binding.FLAG_PARENT_STAYS])
def test_indices_by_the_norm_table_equal_those_of_the_direct_form(B, H, N, d, M, C, flags):
    """avq_forward measures children by norms and products where the grid is large, avq_assign directly: the same indices,
    also where keys and codewords share an offset and the products separate little (one tile per CTA and runs of them)."""
    for offset in (0.0, 4.0, 32.0, 64.0):
        K, Cp, Cc = _offset_inputs(B, H, N, d, M, C, offset, seed=d + M)
        pi, ci = binding.assign(K, Cp, Cc, flags=flags)
        _, _, _, inter = binding.forward(K[:, :, :128].contiguous(), K, K, Cp, Cc, 4, 128, flags=flags, aux=True)
        assert torch.equal(inter["parent_idx"], pi) and torch.equal(inter["child_idx"], ci)


@pytest.mark.parametrize("H,N,d,M", [(24, 1200, 128, 32), (10, 3000, 128, 256), (37, 2001, 64, 96),
                                     (37, 2001, 64, 64)])
def test_eight_children_over_sorted_keys_equal_the_cuda_core_assignment(H, N, d, M):
    """Large grids take eight children by products over keys in the order of their parents: the indices of the CUDA-core
    kernel, which measures every child directly, also with near-ties (an offset) and duplicated children."""
    for offset in (0.0, 32.0):
        K, Cp, Cc = _offset_inputs(1, H, N, d, M, 8, offset, seed=d + M + N)
        pi, ci = binding.assign(K, Cp, Cc)
        pr, cr = binding.assign(K, Cp, Cc, flags=binding.FLAG_SIMT)
        assert torch.equal(pi, pr) and torch.equal(ci, cr)


def test_a_common_offset_costs_little_time():
    """Offsets that bf16 still resolves make the products of the assignment separate less; what they leave open is decided in
    float32 before float64 is asked.  (2.7 times the time of centred inputs with float64 straight away, 1.3 with
    float32 in between.)"""
    def us(offset):
        K, Cp, Cc = _offset_inputs(2, 8, 5000, 128, 96, 8, offset, seed=3, twice=False)
        f = binding.Forward(2, 8, 5000, 5000, 128, 96, 8, 12, 128, flags=binding.FLAG_PARENT_STAYS)
        Y = torch.empty_like(K)
        for _ in range(10):
            f(K, K, K, Cp, Cc, Y)
        times = []
        for _ in range(30):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            f(K, K, K, Cp, Cc, Y)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[len(times) // 2]

    centred, shifted = us(0.0), us(64.0)
    print(f"centred {centred:.1f} us, shifted {shifted:.1f} us")
    assert shifted <= 1.6 * centred


def test_assignment_takes_no_longer_where_every_parent_has_as_many_keys():
    """d = 64, 128 parents of eight children: products over keys in the order of their parents cost 1.5 times as much where the keys
    spread over all parents as where a sixteenth of the parents has all of them (56.5 and 37.4 us); the loop over a key's
    children 1.05 times (50.3 and 47.9)."""
    H, N, M, C = 16, 20000, 128, 8
    _, Cp, Cc = _offset_inputs(1, H, 1, 64, M, C, 0.0, seed=4, twice=False)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)

    def keys(parents):
        at = torch.randint(0, parents * C, (H, N, 1), device="cuda", generator=g).expand(H, N, 64)
        near = Cc.float().view(H, M * C, 64).gather(1, at) + 0.3 * torch.randn(H, N, 64, device="cuda", generator=g)
        return near.to(torch.bfloat16)[None].contiguous()

    def us(K):
        prob = binding.problem(1, H, N, N, 64, M, C, binding.AVQ_BF16, 1.0)
        pi, ci = torch.empty(2, 1, H, N, dtype=torch.int32, device="cuda")
        call = lambda: binding.lib().avq_assign(prob, K.data_ptr(), Cp.data_ptr(), Cc.data_ptr(), pi.data_ptr(), ci.data_ptr(),
                                                binding._raw_stream())
        for _ in range(10):
            assert call() == 0
        times = []
        for _ in range(30):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                call()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e2)
        return sorted(times)[len(times) // 2]

    spread, few = us(keys(M)), us(keys(M // 16))
    print(f"spread {spread:.1f} us, crowded {few:.1f} us")
    assert spread <= 1.2 * few
