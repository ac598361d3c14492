"""Member lists of the gather merge at the edges of their builders: a CTA or a cluster of two, four or eight per head (2048,
4096, 8192 non-pivots), the counting sort for many heads (short and long lists), odd and even slot counts, budgets too large for the
clusters (2700 pivots), lists that leave shared memory (70 000 non-pivots), everything dropped, everything in one slot.  The step is called on its own with hand-made matches."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import inputs

from gpu_util import gpu_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,B,heads", [(1, 241, 2), (31, 242, 2), (2047, 250, 2), (2048, 251, 2), (4096, 241, 2), (8191, 300, 2), (8192, 301, 2),
                                       (9000, 1691, 2), (20000, 2501, 2), (33000, 257, 2), (9000, 2800, 2), (4096, 241, 300), (4097, 300, 300),
                                       (70000, 300, 1), (38500, 300, 2)])
@pytest.mark.parametrize("kind", ["spread", "dropped", "one"])
def test_merge_of_hand_made_matches(E, B, heads, kind):
    rng = np.random.default_rng(E + B)
    U, Hkv, D, L = 1, heads, 128, E + B
    p = O.OracleParams(U, Hkv, Hkv, D, L, 1, B)
    n = min(Hkv, 2)                                                 # (many heads repeat the data of two)
    rep = lambda x: np.ascontiguousarray(np.tile(x, (1, Hkv // n) + (1,) * (x.ndim - 2)))
    k, v = (rep(inputs.round_to_bf16(rng.standard_normal((U, n, L, D)).astype(np.float32))) for _ in range(2))
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in range(n)])[None].astype(np.int32)
    evi = rep(np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32))
    ret = rep(ret)
    match = rep(rng.integers(-1, B, (U, n, E)).astype(np.int32))
    if kind == "dropped":
        match[rep(rng.random((U, n, E)) < 0.9)] = -1
        match[0, -1] = -1
    elif kind == "one":
        match[:] = B - 1
    sim = np.where(match >= 0, rep(rng.random((U, n, E))), 0).astype(np.float32)
    last = slice(Hkv - n, Hkv)                                      # the last heads are compared
    p_n = O.OracleParams(U, n, n, D, L, 1, B)
    ko, vo = O.merge(p_n, k[:, last], v[:, last], ret[:, last], evi[:, last], match[:, last], sim[:, last].astype(np.float64))[:2]
    fp = gpu_params(p, F.BF16)
    g = [torch.zeros((U, Hkv, B, D), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    t = lambda x: torch.from_numpy(x).cuda()
    F.flowmm_merge(fp, to_dev(k, F.BF16), to_dev(v, F.BF16), t(ret), t(evi), t(match), t(sim), g[0], g[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    for got, ref in zip(g, (ko, vo)):
        ref = np.asarray(ref, dtype=np.float64).reshape(U, n, B, D)
        assert np.all(np.abs(got[:, last].float().cpu().numpy() - ref) <= 2e-2 + 1e-2 * np.abs(ref))
        if Hkv > n and kind != "dropped":
            assert torch.equal(got[:, :n], got[:, last])


@pytest.mark.parametrize("dtype,D", [(F.F32, 64), (F.F32, 128), (F.BF16, 64), (F.BF16, 128)])
@pytest.mark.parametrize("E,B,heads", [(1, 300, 1), (32, 257, 2), (33, 249, 40), (1023, 248, 1), (1024, 300, 30), (1025, 300, 2)])
@pytest.mark.parametrize("kind", ["spread", "popular"])
def test_short_lists(dtype, D, E, B, heads, kind):
    """Lists up to 1024 non-pivots are merged straight from the matches: one slot or four per warp, slots of up to 64 members and
    of more, rows of one to two 16-byte vectors per lane."""
    rng = np.random.default_rng(E + B + D)
    L = E + B
    p = O.OracleParams(1, heads, heads, D, L, 1, B)
    k, v = (rng.standard_normal((1, heads, L, D)).astype(np.float32) for _ in range(2))
    if dtype == F.BF16:
        k, v = inputs.round_to_bf16(k), inputs.round_to_bf16(v)
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in range(heads)])[None].astype(np.int32)
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32)
    match = rng.integers(-1, B, (1, heads, E)).astype(np.int32)
    if kind == "popular":                                           # a few slots of 64, 65 and many members
        match[..., : E // 2] = 7
        match[..., E // 2: E // 2 + 65] = B - 1
        match[..., E // 2 + 65: E // 2 + 129] = 0
    sim = np.where(match >= 0, rng.random((1, heads, E)), 0).astype(np.float32)
    ko, vo = O.merge(p, k, v, ret, evi, match, sim.astype(np.float64))[:2]
    g = [torch.zeros((1, heads, B, D), dtype=torch.bfloat16 if dtype == F.BF16 else torch.float32, device="cuda") for _ in range(2)]
    fp = gpu_params(p, dtype)
    ws = F.alloc_workspace(fp)
    t = lambda x: torch.from_numpy(x).cuda()
    F.flowmm_merge(fp, to_dev(k, dtype), to_dev(v, dtype), t(ret), t(evi), t(match), t(sim), g[0], g[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    tol = 1e-2 if dtype == F.BF16 else 1e-5
    for got, ref in zip(g, (ko, vo)):
        ref = np.asarray(ref, dtype=np.float64).reshape(1, heads, B, D)
        assert np.all(np.abs(got.float().cpu().numpy() - ref) <= tol + tol * np.abs(ref))
