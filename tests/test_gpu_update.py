"""avq_codebook_update against the oracle's codebook_update (appendix "Codeword Clustering During Training")."""
import numpy as np
import pytest
import torch

from oracle import avq_oracle as orc
from paper_2607_12789_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _state(wl, seed):
    g = np.random.default_rng(seed)
    H, M, C, d = wl.H, wl.M, wl.C, wl.d
    Np = g.uniform(0.0, 40.0, size=(H, M)).astype(np.float32)
    Nc = g.uniform(0.0, 10.0, size=(H, M, C)).astype(np.float32)
    Np[:, ::7] = 0.0                                             # codes that have never seen a key
    Nc[:, ::5, 1] = 0.0
    Sp = (g.normal(size=(H, M, d)) * 3 * Np[..., None]).astype(np.float32)
    Sc = (g.normal(size=(H, M, C, d)) * 3 * Nc[..., None]).astype(np.float32)
    return Sp, Np, Sc, Nc


@pytest.mark.parametrize("wl,flags", [(synth.C0.with_(B=2, H=2, seed=21), 0),
                                      (synth.C0.with_(B=2, H=2, seed=22, keys_around_parents=True, sigma_k=0.4),
                                       binding.FLAG_PARENT_STAYS),
                                      (synth.C1.with_(B=2, H=3, N=2000, seed=23), 0),
                                      (synth.C3.with_(B=1, H=2, N=3000, seed=24), 0),
                                      (synth.C1.with_(B=2, H=2, N=1500, seed=25, keys_around_parents=True,
                                                      sigma_k=0.45), binding.FLAG_PARENT_STAYS)],
                         ids=["f32", "f32_parent_stays", "bf16_d64", "bf16_d128_M256", "bf16_parent_stays"])
def test_update_matches_the_oracle(wl, flags):
    x = synth.generate(wl)
    Sp, Np, Sc, Nc = _state(wl, wl.seed)
    td = torch.float32 if wl.dtype == "f32" else torch.bfloat16
    dev = lambda a, t=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(t)
    dS = [dev(a) for a in (Sp, Np, Sc, Nc)]
    Cp2, Cc2 = binding.codebook_update(dev(x["K"], td), dev(x["Cp"], td), dev(x["Cc"], td), *dS, 0.9, flags=flags)
    torch.cuda.synchronize()
    ref = orc.codebook_update(x["K"], x["Cp"], x["Cc"], Sp, Np, Sc, Nc, 0.9,
                              parent_stays=bool(flags & binding.FLAG_PARENT_STAYS))
    for got, key in zip(dS, ("Sp", "Np", "Sc", "Nc")):
        np.testing.assert_allclose(got.cpu().numpy(), ref[key], rtol=2e-5, atol=2e-3, err_msg=key)
    assert np.array_equal(dS[1].cpu().numpy() > 0, ref["Np"] > 0)
    # codebooks: fp32 arithmetic on the fp32 path; one bf16 rounding on top of it on the bf16 path.  A child
    # with (almost) no mass divides a residual by a tiny number on both sides, so compare relative to the
    # displacement it can take.
    tol = 2e-3 if wl.dtype == "f32" else 6e-2
    scale_c = 1.0 + np.abs(ref["Cc"])
    assert np.abs(Cp2.float().cpu().numpy() - ref["Cp"]).max() <= tol
    assert (np.abs(Cc2.float().cpu().numpy() - ref["Cc"]) / scale_c).max() <= tol
    if wl.dtype == "f32":
        np.testing.assert_allclose(Cc2.cpu().numpy().mean(axis=2), Cp2.cpu().numpy(), atol=2e-3)


@pytest.mark.parametrize("dtype,B,M,C", [("f32", 4096, 1024, 16), ("bf16", 30000, 256, 8)])
def test_accumulators_beyond_32_gib(dtype, B, M, C):
    """The sums and counts of a call fill more than 2^31 16-byte words: the update and the CUDA-core forward clear and use
    all of them (the workspace is filled with NaN first)."""
    d, Nk = 128, 2
    need = B * M * (1 + C) * (d + 1) * 4
    assert need > 2 ** 35
    if torch.cuda.mem_get_info()[0] < 1.3 * need:
        pytest.skip("needs 48 GB of free device memory")
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    Cp = (3 * torch.randn(1, M, d, device="cuda", generator=g)).to(td)
    Cc = (Cp.float()[:, :, None] + 0.5 * torch.randn(1, M, C, d, device="cuda", generator=g)).to(td)
    pick = torch.randint(0, M * C, (B * Nk,), device="cuda", generator=g)
    K = (Cc.view(M * C, d)[pick].float() + 0.3 * torch.randn(B * Nk, d, device="cuda", generator=g)).to(td).view(B, 1, Nk, d)
    stats = [torch.rand(s, device="cuda", generator=g) for s in ((1, M, d), (1, M), (1, M, C, d), (1, M, C))]
    before = [s.cpu().numpy() for s in stats]
    ws_bytes = binding.lib().avq_codebook_update_workspace_bytes(binding.problem(B, 1, Nk, Nk, d, M, C, binding._dtype_code(K),
                                                                                1.0))
    torch.empty(ws_bytes, dtype=torch.uint8, device="cuda").fill_(255)   # the allocator hands this block out again
    Cp2, Cc2 = binding.codebook_update(K, Cp, Cc, *stats, 0.9)
    host = lambda t: t.float().cpu().numpy()
    ref = orc.codebook_update(host(K).reshape(1, 1, B * Nk, d), host(Cp), host(Cc), *before, 0.9)
    for got, key in zip(stats, ("Sp", "Np", "Sc", "Nc")):
        np.testing.assert_allclose(got.cpu().numpy(), ref[key], rtol=2e-5, atol=2e-3, err_msg=key)
    torch.cuda.empty_cache()
    if dtype == "bf16":
        return
    f = binding.Forward(B, 1, 1, Nk, d, M, C, 4, 1, dtype=td)
    f.workspace.fill_(255)
    Q, V = torch.randn(B, 1, 1, d, device="cuda", generator=g), torch.randn(B, 1, Nk, d, device="cuda", generator=g)
    Y = f(Q, K, V, Cp, Cc)
    f.check()
    for b in (0, B // 2, B - 1):
        one = binding.forward(Q[b:b + 1], K[b:b + 1], V[b:b + 1], Cp, Cc, 4, 1)
        assert (Y[b:b + 1] - one).abs().max().item() <= 1e-5
    del f
    torch.cuda.empty_cache()
