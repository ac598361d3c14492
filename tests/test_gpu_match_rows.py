"""Matching step on the tensor cores with long candidate lists: the token rows are gathered by the non-pivot list.  Numbers of
non-pivots around the edges of its tiles, layouts of K that no tile of consecutive rows could stand for, modalities that change
inside a tile, through flowmm_match (which is handed the lists) and through flowmm_compress_layer (whose selection lays them out).

Tolerance: a similarity is a sum of 128 products of unit vectors' elements in fp32 (its error below 128 2^-24, as the sum of their
magnitudes is at most 1), norms the same, and four cleared mantissa bits below 2^-19 relative: 2e-5 covers them; a match may be any
pivot whose similarity is within that of the best."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import inputs

from gpu_util import gpu_params, run_gpu, to_dev

pytestmark = pytest.mark.gpu
TOL = 2e-5


def _layout(k, layout):
    """k [U, Hkv, L, D] on the device with other strides, the same values."""
    U, H, L, D = k.shape
    if layout == "tokens_first":
        return k.transpose(1, 2).contiguous().transpose(1, 2)
    if layout == "padded":                                            # rows of 136, heads and units with odd gaps (in 16 bytes)
        pad = torch.full((U, H * (L * 136 + 24) + 8), float("nan"), device="cuda", dtype=k.dtype)
        out = pad.as_strided((U, H, L, D), (pad.shape[1], L * 136 + 24, 136, 1))
        out.copy_(k)
        return out
    return k


def _check(k, m, ret, evi, strat, imp, tau, match, sim):
    n = k / np.linalg.norm(k, axis=-1, keepdims=True)
    U, H = k.shape[:2]
    for u in range(U):
        for h in range(H):
            r, e = ret[u, h], evi[u, h]
            cos = n[u, h, e] @ n[u, h, r].T
            gate = np.broadcast_to(imp[u, h, r] <= tau, cos.shape).copy()
            if strat[u] == 0:
                gate &= m[u, e][:, None] == m[u, r][None, :]
            cos = np.where(gate, cos, -np.inf)
            best, got = cos.max(1), match[u, h]
            assert np.array_equal(got < 0, best == -np.inf)
            on = got >= 0
            assert np.all(cos[on, got[on]] > best[on] - TOL)
            assert np.all(np.abs(sim[u, h][on] - cos[on, got[on]]) < TOL)
            assert np.all(sim[u, h][~on] == 0)


@pytest.mark.parametrize("layout", ["dense", "tokens_first", "padded"])
@pytest.mark.parametrize("E", [1, 127, 128, 129, 255, 256, 257, 600, 4500])
def test_lists_of_any_length(E, layout):
    rng = np.random.default_rng(E)
    U, H, B = 2, 3, 230 + E % 7
    L = B + E
    k = inputs.round_to_bf16(rng.standard_normal((U, H, L, 128)).astype(np.float32))
    m = np.stack([np.arange(L) // 300 % 2, rng.random(L) < 0.6]).astype(np.uint8)
    imp = rng.random((U, H, L)).astype(np.float32)
    strat = np.array([0, 1], np.int32)
    perm = np.argsort(rng.random((U, H, L)), axis=-1)
    ret, evi = np.sort(perm[..., :B], -1).astype(np.int32), np.sort(perm[..., B:], -1).astype(np.int32)
    p = O.OracleParams(U, H, H, 128, L, 1, B, tau=0.8, tau_mode=O.TAU_ABS)
    fp = gpu_params(p, F.BF16)
    ws = F.alloc_workspace(fp)
    match = torch.full((U, H, E), -7, dtype=torch.int32, device="cuda")
    sim = torch.full((U, H, E), float("nan"), device="cuda")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    F.flowmm_match(fp, _layout(to_dev(k, F.BF16), layout), dev(imp), dev(m), dev(ret), dev(evi), dev(strat), match, sim, ws)
    assert F.flowmm_last_device_status(ws) == 0
    _check(k.astype(np.float64), m, ret, evi, strat, imp, 0.8, match.cpu().numpy(), sim.cpu().numpy().astype(np.float64))


@pytest.mark.parametrize("U,H,L,B", [(2, 2, 700, 423), (2, 2, 1024, 300), (2, 1, 4096, 1000), (3, 2, 97, 40), (2, 2, 1024, 100), (2, 1, 4096, 224), (2, 1, 1025, 33), (1, 3, 4200, 2100), (3, 1, 9000, 900), (1, 1, 6144, 5000), (40, 1, 6200, 300), (1, 1, 46000, 230)])
def test_selection_lays_the_rows_out(U, H, L, B):
    """One to eight words of 32 positions per warp, more of them in shared memory, a cluster per head, contexts past one chunk, short and
    long candidate lists; runs of a modality and tokens by turns."""
    rng = np.random.default_rng(L)
    q = inputs.round_to_bf16(rng.standard_normal((U, H, 32, 128)).astype(np.float32))
    k = inputs.round_to_bf16(rng.standard_normal((U, H, L, 128)).astype(np.float32))
    m = (np.arange(L)[None] // (100 if U > 1 else 1) % 2 ^ np.arange(U)[:, None] % 2).astype(np.uint8)
    p = O.OracleParams(U, H, H, 128, L, 32, B, tau=2.0, tau_mode=O.TAU_REL, theta=0.5)
    g = run_gpu(p, q, k, k, m, F.BF16)
    n_units = min(U, 3)
    tau = 2.0 * 32 / L
    _check(k[:n_units].astype(np.float64), m, g["retained"].reshape(U, H, B), g["evicted"].reshape(U, H, L - B), g["strategy"],
           g["importance"].reshape(U, H, L), np.float32(tau), g["match"].reshape(U, H, L - B), g["match_sim"].reshape(U, H, L - B))


@pytest.mark.parametrize("H,B,E", [(40, 1300, 1892), (75, 2300, 600), (150, 1100, 300)])
def test_halves_that_sit_items_out(H, B, E):
    """More items than SMs, the last one of a head of one half of 128 rows: the other half's warps are tiles behind or ahead when the
    CTA goes on, with five to nine tiles of candidates and their norms to an item."""
    rng = np.random.default_rng(E)
    U, L = 2, B + E
    k = inputs.round_to_bf16(rng.standard_normal((U, H, L, 128)).astype(np.float32) * np.exp(rng.uniform(-2, 2, (U, H, L, 1))).astype(np.float32))
    m = np.stack([np.arange(L) // 300 % 2, rng.random(L) < 0.3]).astype(np.uint8)
    imp = rng.random((U, H, L)).astype(np.float32)
    strat = np.array([0, 1], np.int32)
    perm = np.argsort(rng.random((U, H, L)), axis=-1)
    ret, evi = np.sort(perm[..., :B], -1).astype(np.int32), np.sort(perm[..., B:], -1).astype(np.int32)
    fp = gpu_params(O.OracleParams(U, H, H, 128, L, 1, B, tau=1.0, tau_mode=O.TAU_ABS), F.BF16)
    ws = F.alloc_workspace(fp)
    match, sim = torch.full((U, H, E), -7, dtype=torch.int32, device="cuda"), torch.full((U, H, E), float("nan"), device="cuda")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    F.flowmm_match(fp, to_dev(k, F.BF16), dev(imp), dev(m), dev(ret), dev(evi), dev(strat), match, sim, ws)
    assert F.flowmm_last_device_status(ws) == 0
    _check(k, m, ret, evi, strat, imp, 1.0, match.cpu().numpy(), sim.cpu().numpy().astype(np.float64))
