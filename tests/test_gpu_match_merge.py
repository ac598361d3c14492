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
