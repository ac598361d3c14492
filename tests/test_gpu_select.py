"""Selection kernel at the edges of its shapes: words of 32 positions, the block sizes (1024, 4096 tokens), contexts that
exceed what fits in shared memory at once (45248 tokens), ties at the threshold, forced windows."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F

from gpu_util import gpu_params, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,B", [(1, 1), (33, 32), (640, 64), (1024, 1), (1025, 1024), (4096, 400), (4097, 211), (33792, 1690),
                                 (45248, 5000), (45249, 77), (100003, 9000)])
@pytest.mark.parametrize("kind", ["spread", "ties", "equal", "window"])
def test_select_against_oracle(L, B, kind):
    rng = np.random.default_rng(L + B)
    imp = np.exp(rng.standard_normal((3, 2, L)) * 2).astype(np.float32)
    if kind == "ties":                                              # few distinct values: the threshold is shared by many
        imp = np.round(imp * 2) / 2
    elif kind == "equal":
        imp[:] = 0.125
    W = min(L, B, 16) if kind == "window" else 1
    p = O.OracleParams(3, 4, 2, 64, L, W, B, keep_window=int(kind == "window"))
    ref_r, ref_e = O.select(p, imp.astype(np.float64))
    fp = gpu_params(p, F.F32)
    r = torch.full((3, 2, B), -9, dtype=torch.int32, device="cuda")
    e = torch.full((3, 2, L - B), -9, dtype=torch.int32, device="cuda")
    F.flowmm_select(fp, torch.from_numpy(imp).cuda(), r, e, F.alloc_workspace(fp))
    assert np.array_equal(r.cpu().numpy(), ref_r)
    assert np.array_equal(e.cpu().numpy(), ref_e)


@pytest.mark.parametrize("heads,L,B", [(600, 512, 60), (600, 513, 60), (600, 640, 64), (600, 1001, 1000), (600, 1024, 200), (160, 257, 40), (160, 1024, 100),
                                       (160, 1025, 100), (160, 4096, 300), (147, 256, 40), (147, 257, 40), (147, 1025, 100), (147, 4096, 300)])
@pytest.mark.parametrize("kind", ["spread", "ties", "equal", "window"])
def test_many_heads(heads, L, B, kind):
    """More heads than four blocks per SM (blocks of 128 threads between 512 and 1024 positions), than one per SM, and one fewer than
    SMs (twice the warps from 257 positions on); and, with the candidates laid out by the same launch, the matches of the separate step."""
    W = 32
    gen = torch.Generator(device="cuda").manual_seed(L + B)
    imp = torch.exp(torch.randn((1, heads, L), generator=gen, device="cuda") * 2)
    if kind == "ties":
        imp = (imp * 2).round() / 2
    elif kind == "equal":
        imp[:] = 0.125
    p = O.OracleParams(1, heads, heads, 128, L, W, B, keep_window=int(kind == "window"), theta=0.3, tau=2.0, tau_mode=O.TAU_REL)
    ref_r, ref_e = O.select(p, imp.cpu().numpy().astype(np.float64))
    fp = gpu_params(p, F.BF16)
    r = torch.full((1, heads, B), -9, dtype=torch.int32, device="cuda")
    e = torch.full((1, heads, L - B), -9, dtype=torch.int32, device="cuda")
    F.flowmm_select(fp, imp, r, e, F.alloc_workspace(fp))
    assert np.array_equal(r.cpu().numpy(), ref_r)
    assert np.array_equal(e.cpu().numpy(), ref_e)
    q, k = (torch.randn((1, heads, n, 128), generator=gen, device="cuda").bfloat16() for n in (W, L))
    m = (torch.arange(L, device="cuda") % 70 < 50).to(torch.uint8)[None]
    out = F.compress_layer_alloc(fp, q, k, k, m)
    match, sim = torch.full_like(out["match"], -9), torch.zeros_like(out["match_sim"])
    F.flowmm_match(fp, k, out["importance"], m, out["retained"], out["evicted"], out["strategy"], match, sim, F.alloc_workspace(fp))
    assert torch.equal(match, out["match"]) and torch.equal(sim, out["match_sim"])


@pytest.mark.parametrize("L,B", [(6143, 600), (6144, 600), (6145, 601), (8192, 8000), (33792, 1690), (45249, 77)])
@pytest.mark.parametrize("U", [1, 18, 20])
@pytest.mark.parametrize("kind", ["spread", "ties"])
def test_select_by_clusters_and_by_blocks(L, B, U, kind):
    """Long contexts with few heads (a cluster of CTAs for each, the last CTA's part short or empty) and with many (one block)."""
    rng = np.random.default_rng(L + U)
    imp = np.exp(rng.standard_normal((U, 2, L)) * 2).astype(np.float32)
    if kind == "ties":
        imp = np.round(imp * 2) / 2
    p = O.OracleParams(U, 4, 2, 64, L, 16, B, keep_window=1)
    ref_r, ref_e = O.select(p, imp.astype(np.float64))
    fp = gpu_params(p, F.F32)
    r = torch.full((U, 2, B), -9, dtype=torch.int32, device="cuda")
    e = torch.full((U, 2, L - B), -9, dtype=torch.int32, device="cuda")
    F.flowmm_select(fp, torch.from_numpy(imp).cuda(), r, e, F.alloc_workspace(fp))
    assert np.array_equal(r.cpu().numpy(), ref_r)
    assert np.array_equal(e.cpu().numpy(), ref_e)


@pytest.mark.parametrize("L,B", [(290, 193), (7000, 130), (9000, 700), (2000, 225), (46000, 300), (6000, 4096), (6000, 4097), (12000, 9000),
                                 (3000, 512), (3000, 513)])
def test_fused_preparation_equals_the_steps(L, B):
    """The candidate layout written by the selection launch of flowmm_compress_layer against the one flowmm_match makes
    from the lists: same matches, bit for bit (short lists, long lists, a context of more than one chunk)."""
    rng = np.random.default_rng(L)
    p = O.OracleParams(2, 2, 1, 128, L, 32, B, theta=0.3, tau=2.0, tau_mode=O.TAU_REL)
    q, k, v = (rng.standard_normal(s).astype(np.float32) for s in ((2, 2, 32, 128), (2, 1, L, 128), (2, 1, L, 128)))
    m = (np.arange(L) % 700 < 500).astype(np.uint8)[None].repeat(2, 0)
    got = run_gpu(p, q, k, v, m, F.BF16)
    fp = gpu_params(p, F.BF16)
    dev = lambda key, dt: torch.from_numpy(got[key]).to(dt).cuda()
    match = torch.full((2, 1, L - B), -9, dtype=torch.int32, device="cuda")
    sim = torch.zeros((2, 1, L - B), device="cuda")
    F.flowmm_match(fp, torch.from_numpy(k).cuda().bfloat16(), dev("importance", torch.float32), torch.from_numpy(m).cuda(),
                   dev("retained", torch.int32), dev("evicted", torch.int32), dev("strategy", torch.int32), match, sim, F.alloc_workspace(fp))
    assert np.array_equal(match.cpu().numpy(), got["match"])
    assert np.array_equal(sim.cpu().numpy().astype(np.float64), got["match_sim"])
