"""Scoring step on the tensor cores (two passes) against the oracle where its ways through a tile part: chunks of 32 keys of one
modality or of both, a modality that changes inside a word, at a word or at a tile, windows of both modalities, ends of the
prompt inside a chunk, one to four tiles of proxy rows, and row statistics of so many key chunks that a launch joins them.

Tolerance: an exponential is within 4e-6 of its value (the polynomial quarter; exp2.approx is closer) and enters numerator and
normaliser, logits of a few units in fp32 add less than 1e-6, sums of fp32 parts another 1e-6: importances within 1e-5 relative, a
row's share of its mass within 1e-5 of the row's mass 1, a head's mass of W rows within 1e-5 W."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import inputs

from gpu_util import gpu_params, to_dev

pytestmark = pytest.mark.gpu

PATTERNS = {
    "one": lambda rng, L: np.ones(L),
    "none": lambda rng, L: np.zeros(L),
    "every_other": lambda rng, L: np.arange(L) % 2,
    "random": lambda rng, L: rng.random(L) < 0.8,
    "run_in_word": lambda rng, L: (np.arange(L) >= 41) & (np.arange(L) < L - 75),
    "runs_of_words": lambda rng, L: np.arange(L) // 32 % 2,
    "runs_of_tiles": lambda rng, L: np.arange(L) // 256 % 2,
    "window_of_both": lambda rng, L: np.arange(L) >= L - 20,
}


def _check(rng, U, Hq, Hkv, L, W, modality):
    p = O.OracleParams(U, Hq, Hkv, 128, L, W, 1)
    q = inputs.round_to_bf16(rng.standard_normal((U, Hq, W, 128)).astype(np.float32))
    k = inputs.round_to_bf16(rng.standard_normal((U, Hkv, L, 128)).astype(np.float32))
    m = np.ascontiguousarray(modality, dtype=np.uint8)
    imp, cross, _ = O.score(p, q, k, m)
    fp = gpu_params(p, F.BF16)
    g_imp = torch.full((U, Hkv, L), float("nan"), device="cuda")
    g_cross = torch.full((U, Hq), float("nan"), device="cuda")
    ws = F.alloc_workspace(fp)
    F.flowmm_score(fp, to_dev(q, F.BF16), to_dev(k, F.BF16), torch.from_numpy(m).cuda(), g_imp, g_cross, ws)
    assert F.flowmm_last_device_status(ws) == 0
    g_imp, g_cross = g_imp.cpu().numpy().astype(np.float64), g_cross.cpu().numpy().astype(np.float64)
    assert np.abs(g_imp / imp - 1).max() < 1e-5
    assert np.abs(g_cross - cross).max() < 1e-5 * W
    if m.min() == m.max():
        assert np.all(g_cross == 0.0)


@pytest.mark.parametrize("pattern", sorted(PATTERNS))
@pytest.mark.parametrize("G,W,L", [(7, 32, 1471), (7, 64, 641), (3, 128, 256), (8, 128, 289), (4, 32, 2049)])
def test_modality_patterns(pattern, G, W, L):
    rng = np.random.default_rng(L + G)
    _check(rng, 2, 2 * G, 2, L, W, np.stack([PATTERNS[pattern](rng, L), rng.random(L) < 0.5]))


@pytest.mark.parametrize("L", [64, 65, 95, 96, 97, 255, 257, 511, 513])
def test_ends_of_the_prompt(L):
    rng = np.random.default_rng(L)
    _check(rng, 3, 4, 2, L, 64, rng.random((3, L)) < 0.5)


@pytest.mark.parametrize("U,G,W,L", [(37, 12, 64, 600), (150, 3, 32, 200), (299, 2, 64, 257), (5, 4, 64, 2600), (1, 7, 32, 5000)])
def test_runs_of_tiles_across_heads(U, G, W, L):
    """Runs that hold many heads, end inside heads, and heads spread over many runs, with one to three tiles of proxy rows."""
    rng = np.random.default_rng(U)
    _check(rng, U, G, 1, L, W, np.arange(L)[None] // 100 % 2 ^ rng.integers(0, 2, (U, 1)))


@pytest.mark.parametrize("L", [4096, 4097, 9001])
def test_many_key_chunks_of_one_head(L):
    rng = np.random.default_rng(L)
    _check(rng, 1, 8, 1, L, 64, np.arange(L)[None] // 1000 % 2)


@pytest.mark.parametrize("U,G,W,L", [(74, 2, 128, 256), (75, 2, 128, 256), (74, 2, 128, 257), (18, 8, 128, 200), (19, 8, 128, 200),
                                     (148, 5, 32, 128), (149, 5, 32, 128), (49, 5, 32, 384), (50, 5, 32, 385), (2, 5, 32, 129)])
def test_items_of_one_half_and_of_two(U, G, W, L):
    """Both sides of the lines at which either pass goes from items of 128 proxy rows or keys to items of 256."""
    rng = np.random.default_rng(U * L)
    _check(rng, U, G, 1, L, W, np.arange(L)[None] // 50 % 2 ^ rng.integers(0, 2, (U, 1)))


@pytest.mark.parametrize("G,W", [(2, 64), (7, 32), (7, 64)])
@pytest.mark.parametrize("L", [513, 640])
def test_runs_of_half_items(G, W, L):
    """112 heads of five halves of an item: the second pass gives all warps of a CTA one half at a time, four to a CTA, in each of its
    three shapes."""
    rng = np.random.default_rng(G * W + L)
    _check(rng, 112, G, 1, L, W, np.arange(L)[None] // 50 % 2 ^ rng.integers(0, 2, (112, 1)))


def test_sums_over_many_proxy_rows():
    """A key of the window that one proxy row gives all of its mass and 1023 others 2.5e-8 each: added to the one, one by one, they would
    vanish (half of them share its sum: 1.3e-5).  Exponentials within 2^-22, their arguments (up to 26) within 2e-6, sums of 32 by fours."""
    L, W, G = 300, 128, 8
    q, k = np.zeros((1, G, W, 128), np.float32), np.zeros((1, 1, L, 128), np.float32)
    q[..., 0], q[..., 2] = 1, 1
    q[0, 0, 0, 0], q[0, 0, 0, 1] = 0, 1
    k[0, 0, 1:, 2] = -1024                                          # (logit -90)
    k[0, 0, L - W, 0], k[0, 0, L - W, 2] = -198, 0                  # (logit -17.5)
    k[0, 0, 0, 1], k[0, 0, L - W, 1] = -1024, 0
    q, k = inputs.round_to_bf16(q), inputs.round_to_bf16(k)
    p = O.OracleParams(1, G, 1, 128, L, W, 1)
    m = np.zeros((1, L), np.uint8)
    imp = O.score(p, q, k, m)[0][0, 0, L - W]
    fp = gpu_params(p, F.BF16)
    g_imp, g_cross = torch.zeros((1, 1, L), device="cuda"), torch.zeros((1, G), device="cuda")
    ws = F.alloc_workspace(fp)
    F.flowmm_score(fp, to_dev(q, F.BF16), to_dev(k, F.BF16), torch.from_numpy(m).cuda(), g_imp, g_cross, ws)
    assert F.flowmm_last_device_status(ws) == 0
    assert imp > 0.125 * (1 + 2e-5) and abs(float(g_imp[0, 0, L - W]) / imp - 1) < 1e-6


@pytest.mark.parametrize("pattern", ["random", "run_in_word", "window_of_both"])
@pytest.mark.parametrize("G,W,L", [(3, 32, 97), (4, 32, 1024), (4, 32, 1025), (4, 32, 4096), (4, 32, 4097), (7, 32, 1471), (8, 32, 2048), (8, 32, 2049),
                                   (3, 128, 256), (7, 64, 641), (8, 64, 1024), (8, 64, 1025), (4, 32, 791),
                                   (2, 32, 97), (2, 32, 2048), (2, 32, 2049), (1, 64, 641)])
def test_few_heads_and_many_of_the_same(G, W, L, pattern):
    """One unit, whose heads are shared by clusters of one to eight CTAs of one, two or four key tiles (up to the longest prompt that
    one to four tiles of proxy rows leave room for); eight of it, for which some sizes of clusters do not find room; and sixty and eighty
    times that unit, which take the two passes (sixty with more than one CTA to a head)."""
    rng = np.random.default_rng(L + G)
    modality = PATTERNS[pattern](rng, L)[None]
    p = O.OracleParams(1, 2 * G, 2, 128, L, W, 1)
    q, k = (inputs.round_to_bf16(rng.standard_normal(s).astype(np.float32)) for s in ((1, 2 * G, W, 128), (1, 2, L, 128)))
    m = np.ascontiguousarray(modality, dtype=np.uint8)
    imp, cross, _ = O.score(p, q, k, m)
    qd, kd, md = to_dev(q, F.BF16), to_dev(k, F.BF16), torch.from_numpy(m).cuda()
    for U in (1, 8, 60, 80):
        fp = F.Params(U, 2 * G, 2, 128, L, W, 1)
        g_imp, g_cross = torch.full((U, 2, L), float("nan"), device="cuda"), torch.full((U, 2 * G), float("nan"), device="cuda")
        ws = F.alloc_workspace(fp)
        F.flowmm_score(fp, qd.repeat(U, 1, 1, 1), kd.repeat(U, 1, 1, 1), md.repeat(U, 1), g_imp, g_cross, ws)
        assert F.flowmm_last_device_status(ws) == 0
        for u in (0, U - 1):
            assert np.abs(g_imp[u].double().cpu().numpy() / imp[0] - 1).max() < 1e-5
            assert np.abs(g_cross[u].double().cpu().numpy() - cross[0]).max() < 1e-5 * W
