"""GPU parity of the CUDA-core kernels (float32 path and AVQ_FLAG_SIMT) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import avq_oracle as orc
from paper_2607_12789_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu
SIMT, STAYS = binding.FLAG_SIMT, binding.FLAG_PARENT_STAYS


def test_c0_tiny_f32_full_parity():
    rep = parity.full_parity(synth.C0)
    assert rep["max_abs"] <= 1e-4
    assert rep["stay_count"] == 0


@pytest.mark.parametrize("P", [0, 1, 5, 16])
def test_c0_endpoints_and_other_P(P):
    parity.full_parity(synth.C0, P=P)


def test_ragged_shapes_f32():
    wl = synth.Workload("ragged", B=2, H=3, N=333, d=36, M=11, C=3, P=4, block_q=50, dtype="f32", seed=21,
                        alpha=0.5)
    x = synth.generate(wl)
    x["Q"] = np.ascontiguousarray(x["Q"][:, :, :171])          # Nq != Nk, both ragged
    parity.full_parity(wl, x=x)


def test_parent_stays_f32():
    wl = synth.C0.with_(seed=5, H=2)
    x = synth.generate(wl)
    g = np.random.default_rng(0)
    for h in range(2):                                           # every other key hugs a parent: it stays
        near = x["Cp"][h][g.integers(0, 16, 128)] + 0.05 * g.standard_normal((128, 64)).astype(np.float32)
        x["K"][0, h, ::2] = near
    rep = parity.full_parity(wl, flags=STAYS, parent_stays=True, x=x)
    assert 200 <= rep["stay_count"] < 2 * 256                   # a real mixture of stayed and moved keys


def test_bf16_inputs_through_cuda_cores():
    wl = synth.C1.with_(B=1, H=3, N=512)
    rep = parity.full_parity(wl, flags=SIMT)
    assert rep["empty_parents"] > 0
    wl = synth.C2.with_(B=1, H=2, N=640)
    parity.full_parity(wl, flags=SIMT)


def test_exact_ties_resolve_to_lowest_index():
    g = np.random.default_rng(0)
    d, M, C = 16, 8, 4
    base = (np.clip(np.round(g.normal(size=(4, d)) * 4), -8, 8) / 4).astype(np.float32)   # exact in bf16
    Cp = np.stack([base[0], base[1], base[1], base[2], base[0], base[3], base[3], base[3]])[None]
    Cc = np.repeat(Cp[:, :, None, :], C, axis=2).copy()
    Cc[0, :, 2:] += 0.25                                          # children 0,1 equal; 2,3 equal
    K = np.concatenate([Cp[0], Cp[0] + 0.125, 0.5 * (Cp[0, [0]] + Cp[0, [1]])])[None, None]
    ref = orc.assign_head(K[0, 0], Cp[0], Cc[0])
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    for dt, fl in ((torch.float32, 0), (torch.bfloat16, SIMT)):
        pi, ci = binding.assign(t(K).to(dt), t(Cp).to(dt), t(Cc).to(dt), flags=fl)
        assert np.array_equal(pi.cpu().numpy()[0, 0], ref["parent_idx"])
        assert np.array_equal(ci.cpu().numpy()[0, 0], ref["child_idx"])
    assert ref["parent_idx"][:8].tolist() == [0, 1, 1, 3, 0, 5, 5, 5]
    assert (ref["parent_margin"][:8] == 0).sum() >= 6


def test_standalone_stages_match_forward_intermediates():
    wl = synth.C0.with_(H=2, seed=3)
    x = synth.generate(wl)
    dv = parity.to_device(x, "f32")
    pi, ci = binding.assign(dv["K"], dv["Cp"], dv["Cc"])
    Vp, n_p, Vc, n_c = binding.aggregate(dv["V"], pi, ci, wl.M, wl.C)
    _, _, _, inter = binding.forward(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q, aux=True)
    assert torch.equal(pi, inter["parent_idx"]) and torch.equal(ci, inter["child_idx"])
    assert torch.equal(n_p, inter["np"]) and torch.equal(n_c, inter["nc"])
    assert torch.allclose(Vp, inter["Vp"], atol=1e-4) and torch.allclose(Vc, inter["Vc"], atol=1e-4)
    assert float(n_p.sum()) == wl.B * wl.H * wl.N


def test_forward_host_matches_device_call():
    wl = synth.C0
    x = synth.generate(wl)
    dv = parity.to_device(x, "f32")
    f = binding.Forward(1, 1, 256, 256, 64, 16, 4, 2, 64, dtype=torch.float32)
    Y = f(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"])
    hq, hk, hv = (torch.from_numpy(x[k]).pin_memory() for k in "QKV")
    hy = torch.empty_like(hq).pin_memory()
    dq, dk, dv_, dy = (torch.empty_like(dv["Q"]) for _ in range(4))
    f.host(hq, hk, hv, dv["Cp"], dv["Cc"], hy, dq, dk, dv_, dy)
    torch.cuda.synchronize()
    f.check()
    assert torch.allclose(hy, Y.cpu(), atol=1e-6)


def test_correcting_form_matches_the_oracle_and_the_masked_form_on_recentred_codebooks():
    """AVQ_FLAG_CORRECTING (Algorithm 2's child pass as printed) on the CUDA-core kernels.  float32, re-centred
    children: equal to the oracle's correcting form and (the constraint holds to fp32 rounding) to the default
    masked form.  bfloat16 codebooks: rounding breaks parent = mean(children) by an ulp, so the kernel is
    compared with the oracle's correcting form on the same rounded codebooks, and its distance from the masked
    form is what the variant costs in accuracy."""
    wl = synth.C0.with_(H=2, seed=33, recenter_children=True)
    x = synth.generate(wl)
    dv = parity.to_device(x, "f32")
    args = (dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q)
    Yc = binding.forward(*args, scale=wl.scale, flags=binding.FLAG_CORRECTING)
    Ym = binding.forward(*args, scale=wl.scale)
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, wl.block_q, wl.scale, form="correcting")
    assert np.abs(Yc.cpu().numpy() - ref["Y"]).max() <= 1e-4
    assert (Yc - Ym).abs().max().item() <= 1e-4
    wl = synth.C1.with_(B=1, H=2, N=512, seed=34, recenter_children=True)
    x = synth.generate(wl)
    dv = parity.to_device(x, "bf16")
    args = (dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], wl.P, wl.block_q)
    Yc = binding.forward(*args, scale=wl.scale, flags=binding.FLAG_CORRECTING | SIMT)
    Ym = binding.forward(*args, scale=wl.scale, flags=SIMT)
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, wl.block_q, wl.scale, form="correcting")
    assert np.abs(Yc.float().cpu().numpy() - ref["Y"]).max() <= 2e-2
    dev = (Yc.float() - Ym.float()).abs().max().item()
    print(f"correcting vs masked form, bf16-rounded re-centred codebooks: max-abs {dev:.3e}")
    assert dev <= 0.25


@pytest.mark.parametrize("d,M,C,P,bq,N", [(4, 1, 1, 1, 1, 70), (64, 64, 4, 8, 65, 131), (68, 65, 5, 7, 129, 300),
                                          (128, 130, 16, 3, 200, 450), (132, 70, 2, 70, 64, 200),
                                          (256, 33, 3, 0, 100, 210), (64, 300, 4, 20, 128, 256)])
def test_tile_edges_of_the_register_tiled_kernels(d, M, C, P, bq, N):
    """64-key, 64-codeword and 64- / 128-row tiles: one element past and short of a tile, several row tiles per
    query block, every head-dimension variant, logits kept in shared memory and recomputed."""
    wl = synth.Workload("edges", B=1, H=2, N=N, d=d, M=M, C=C, P=P, block_q=bq, dtype="f32", seed=70 + d, alpha=0.6)
    parity.full_parity(wl)
    x = synth.generate(wl)
    dv = parity.to_device(x, "f32")
    if P in (0, M) or M < 64:
        return
    # importance over tiles of 32 parents (narrower than a codeword tile)
    _, topp, imp = binding.forward_tiled(dv["Q"], dv["K"], dv["V"], dv["Cp"], dv["Cc"], P, bq, 32, scale=wl.scale)
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], P, bq, wl.scale, form="factorised", tile_m=32)
    parity.compare_selection(dict(selected=topp.cpu().numpy(), importance=imp.cpu().numpy()), ref)


@pytest.mark.parametrize("dtype,flags", [("f32", 0), ("bf16", SIMT)])
def test_logits_beyond_the_range_of_fp32_weigh_nothing(dtype, flags):
    """The first 64 parents, a whole codeword tile, and their children have logits of -1e39, -inf in fp32: their weights
    are 0 as long as any other codeword holds a key."""
    wl = synth.Workload("neg", B=1, H=2, N=300, d=64, M=130, C=3, P=9, block_q=128, dtype=dtype, seed=91, alpha=0.8)
    x = synth.generate(wl)
    for k in ("Q", "K", "Cp", "Cc"):
        x[k][..., 0] = 0.0
    x["Q"][..., 0] = 1e31
    x["Cp"][:, :64, 0] = x["Cc"][:, :64, :, 0] = -1e9
    x["K"][:, :, ::2, 0] = -1e9                                  # every other key belongs to one of them
    x = {k: (synth.round_to_bf16(v) if dtype == "bf16" else v) for k, v in x.items()}
    gpu = parity.gpu_forward(wl, x, flags=flags)
    ref = orc.forward(x["Q"], x["K"], x["V"], x["Cp"], x["Cc"], wl.P, wl.block_q, wl.scale, form="factorised")
    assert (ref["np"][..., :64].sum(-1) == 150).all() and (ref["importance"][..., :64] == 0).all()
    same, _ = parity.compare_selection(gpu, ref)
    parity.compare_output(gpu["Y"], ref["Y"], dtype, np.repeat(same, wl.block_q, axis=-1)[..., :wl.N])


@pytest.mark.parametrize("dtype,d,M,C,P,bq,flags", [("bf16", 128, 193, 1, 13, 128, SIMT), ("f32", 4, 701, 1, 1, 64, 0)])
def test_logits_that_just_miss_shared_memory_are_recomputed(dtype, d, M, C, P, bq, flags):
    """One-wave grids keep a block's logits in shared memory if all of it fits a CTA: at these sizes it exceeds the limit
    by less than the kernel's own counters take.  The call answers, and so does an ordinary one behind it."""
    wl = synth.Workload("limit", B=1, H=1, N=300, d=d, M=M, C=C, P=P, block_q=bq, dtype=dtype, seed=92, alpha=0.8)
    parity.full_parity(wl, flags=flags)
    parity.full_parity(synth.C0)


def test_threads_with_problems_of_different_size_do_not_disturb_each_other():
    """Eight threads, each with its own stream and workspace, launch the same kernels with small and large shared-memory
    needs: no call fails, and every output is what the call gives alone."""
    import threading

    def problem(i):
        g = torch.Generator(device="cuda")
        g.manual_seed(i)
        r = lambda *s: torch.randn(*s, device="cuda", generator=g)
        M, d = (16, 300, 64, 500)[i % 4], (64, 36)[i // 4]
        f = binding.Forward(1, 1, 200, 200, d, M, 2, 2, 64, dtype=torch.float32)
        return f, (r(1, 1, 200, d), r(1, 1, 200, d), r(1, 1, 200, d), r(1, M, d), r(1, M, 2, d))

    problems = [problem(i) for i in range(8)]
    alone = [f(*args) for f, args in problems]
    torch.cuda.synchronize()
    failed, last = [], [None] * 8

    def work(i):
        f, args = problems[i]
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(600):
                try:
                    last[i] = f(*args)
                except binding.AvqError as e:
                    failed.append(e)
        s.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for y, y0 in zip(last, alone):
        assert (y - y0).abs().max().item() <= 1e-5               # (the value sums are added in any order)


@pytest.mark.parametrize("d,M,C,P,bq,N,stays", [(4, 33, 2, 5, 1, 70, False), (36, 65, 3, 7, 50, 131, False), (68, 130, 5, 9, 129, 300, False),
                                                (132, 65, 2, 65, 64, 200, False), (256, 33, 4, 0, 100, 210, False),
                                                (64, 64, 4, 8, 64, 200, False), (128, 130, 16, 3, 200, 450, True),
                                                (36, 33, 4, 6, 50, 260, True)])
def test_tile_edges_with_bf16_inputs(d, M, C, P, bq, N, stays):
    """As above for bfloat16 on the CUDA cores: products by 16 x 8 x 16 tiles (head dimensions that are no multiple of 16,
    padded rows and columns), every row-tile variant, both child rules."""
    wl = synth.Workload("edges16", B=1, H=2, N=N, d=d, M=M, C=C, P=P, block_q=bq, dtype="bf16", seed=170 + d, alpha=0.6)
    x = synth.generate(wl)
    if stays:                                                    # every other key hugs a parent: it stays
        x["K"][:, :, ::2] = synth.round_to_bf16(x["Cp"][None, :, np.arange(0, N, 2) % M] + np.float32(0.03))
    rep = parity.full_parity(wl, flags=SIMT | (STAYS if stays else 0), parent_stays=stays, x=x)
    assert not stays or 0.8 * N < rep["stay_count"] < 1.2 * N
