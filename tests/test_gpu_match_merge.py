"""Matching and merge in one launch (the fused call with many heads of few pivots) against the two steps one after the
other: the same matches and the same bits of the compressed cache, as both take the products in the same order."""
import pytest
import torch

from paper_2511_05534_b200 import binding as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,L,B,kw", [
    (75, 33, 1, {}), (80, 129, 1, {}), (80, 200, 17, {}), (148, 256, 16, {}),   # the fewest heads, one per CTA; one to five steps of 128 tokens
    (80, 1290, 64, {}), (90, 300, 64, dict(tau=0.0)),               # many steps; no candidate
    (180, 385, 33, {}), (310, 400, 32, dict(merge_mode=F.MERGE_MEAN)), (400, 640, 64, {}), (200, 513, 48, dict(keep_window=1)),   # heads by turns
    (80, 640, 65, {}), (74, 640, 64, {}), (310, 384, 64, {}), (160, 640, 64, {}),   # past the most slots; too few heads or steps: two launches
])
@pytest.mark.parametrize("flow", [1, 2])
def test_one_launch_equals_the_steps(heads, L, B, kw, flow):
    W = 32
    args = dict(theta=0.4, tau=1.5, tau_mode=F.TAU_REL, flow_mode=flow)
    args.update(kw)
    gen = torch.Generator(device="cuda").manual_seed(heads * L + B)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    q, k, v = draw(1, heads, W, 128), draw(1, heads, L, 136)[..., :128], draw(1, heads, L, 128)     # (K's rows apart)
    m = ((torch.arange(L, device="cuda") + 13) % 190 > 40).to(torch.uint8)[None]
    p = F.Params(1, heads, heads, 128, L, W, B, **args)
    full = F.compress_layer_alloc(p, q, k, v, m)
    assert F.flowmm_last_device_status(full["ws"]) == 0
    match, sim = torch.full_like(full["match"], -9), torch.zeros_like(full["match_sim"])
    ws = F.alloc_workspace(p)
    F.flowmm_match(p, k, full["importance"], m, full["retained"], full["evicted"], full["strategy"], match, sim, ws)
    k_out, v_out = torch.zeros_like(full["k_out"]), torch.zeros_like(full["v_out"])
    F.flowmm_merge(p, k, v, full["retained"], full["evicted"], match, sim, k_out, v_out, ws)
    assert torch.equal(match, full["match"]) and torch.equal(sim, full["match_sim"])
    assert torch.equal(k_out, full["k_out"]) and torch.equal(v_out, full["v_out"])
    # nobody asks for the matches; output rows apart; a workspace that has been used
    k2, v2 = (torch.zeros((1, heads, B, 144), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for _ in range(3):
        F.flowmm_compress_layer(p, q, k, v, m, k2[..., :128], v2[..., :128], ws)
    assert torch.equal(k2[..., :128], k_out) and torch.equal(v2[..., :128], v_out)
    assert not k2[..., 128:].any() and not v2[..., 128:].any()
    assert F.flowmm_last_device_status(ws) == 0


@pytest.mark.parametrize("U,Hkv,G,L,B", [(20, 4, 2, 300, 48), (40, 8, 1, 400, 33), (3, 32, 1, 700, 64)])
def test_units_of_both_strategies_and_matches_alone(U, Hkv, G, L, B):
    """Several units, whose modalities and strategies differ; of the matches' two tensors both, either or none asked for."""
    W = 32
    gen = torch.Generator(device="cuda").manual_seed(U * L)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    q, k, v = draw(U, Hkv * G, W, 128), draw(U, Hkv, L, 128), draw(U, Hkv, L, 128)
    share = torch.linspace(0.05, 0.95, U, device="cuda")[:, None]
    m = (torch.rand((U, L), generator=gen, device="cuda") < share).to(torch.uint8)
    p = F.Params(U, Hkv * G, Hkv, 128, L, W, B, theta=0.4, tau=1.5, tau_mode=F.TAU_REL)
    rho = F.compress_layer_alloc(p, q, k, v, m)["rho"]
    p = F.Params(U, Hkv * G, Hkv, 128, L, W, B, theta=float(rho.sort().values[U // 2 - 1:U // 2 + 1].mean()), tau=1.5, tau_mode=F.TAU_REL)
    full = F.compress_layer_alloc(p, q, k, v, m)
    assert F.flowmm_last_device_status(full["ws"]) == 0 and 0 < int(full["strategy"].sum()) < U
    match, sim = torch.full_like(full["match"], -9), torch.zeros_like(full["match_sim"])
    ws = F.alloc_workspace(p)
    F.flowmm_match(p, k, full["importance"], m, full["retained"], full["evicted"], full["strategy"], match, sim, ws)
    k_out, v_out = torch.zeros_like(full["k_out"]), torch.zeros_like(full["v_out"])
    F.flowmm_merge(p, k, v, full["retained"], full["evicted"], match, sim, k_out, v_out, ws)
    assert torch.equal(match, full["match"]) and torch.equal(sim, full["match_sim"])
    assert torch.equal(k_out, full["k_out"]) and torch.equal(v_out, full["v_out"])
    for asked in ((), ("match",), ("match_sim",)):
        out = {key: torch.full_like(full[key], -9) for key in ("k_out", "v_out") + asked}
        F.flowmm_compress_layer(p, q, k, v, m, out["k_out"], out["v_out"], ws, **{key: out[key] for key in asked})
        assert F.flowmm_last_device_status(ws) == 0
        assert all(torch.equal(out[key], full[key]) for key in out)
