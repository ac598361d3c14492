"""Merge of sorted lists by windows of rows: slots of chosen numbers of members (none, the most that stay whole, one more, several
pieces) at chosen places of a window, windows of 16, 32 and 64 rows, taken with a stride or drawn from the counter,
pieces of long slots as items of their own and spread over the windows, every row width, and output layouts with gaps.
The values let one lost or doubled member be seen (test_merge_reference.py)."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F

from gpu_util import gpu_params, merge_reference, small_integers, to_dev

pytestmark = pytest.mark.gpu


def _members(pattern, B, rng):
    """Members of each slot."""
    n = rng.integers(0, 4, B)
    edges = [63, 64, 65, 127, 128, 129, 130, 191, 192, 193, 257, 640]
    if pattern == "edges_first":
        n[: len(edges)] = edges
    elif pattern == "edges_apart":                                  # every one at another place of its window
        n[7:7 + 17 * len(edges):17] = edges
    elif pattern == "edges_last":
        n[B - len(edges):] = edges
    elif pattern == "alternate":
        n[:] = 0
        n[5:65:2] = np.tile([65, 15, 64, 129, 1], 6)
    return n


@pytest.mark.parametrize("dtype,D", [(F.BF16, 128), (F.BF16, 64), (F.F32, 64), (F.F32, 128)])
@pytest.mark.parametrize("heads", [1, 12, 90])                     # windows of 16, of 32 with pieces of their own, of 32 with pieces spread
@pytest.mark.parametrize("pattern", ["edges_first", "edges_apart", "edges_last", "alternate"])
def test_slots_of_chosen_sizes(pattern, heads, dtype, D):
    rng = np.random.default_rng(D + heads)
    B = 700
    n = _members(pattern, B, rng)
    dropped = 150
    E = int(n.sum()) + dropped
    L = E + B
    if E <= 1024:
        pytest.skip("short list")
    k, v = (small_integers(rng, (1, 1, L, D)) for _ in range(2))
    ret = np.sort(rng.choice(L, B, replace=False))
    evi = np.setdiff1d(np.arange(L), ret)
    match = np.concatenate([np.repeat(np.arange(B), n), np.full(dropped, -1)])
    rng.shuffle(match)
    sim = np.where(match >= 0, rng.random(E), 0).astype(np.float32)
    ret, evi, match = (x.astype(np.int32)[None, None] for x in (ret, evi, match))
    sim = sim[None, None]
    rep = lambda x: torch.from_numpy(np.ascontiguousarray(np.repeat(x, heads, 1))).cuda()
    lists = [rep(x) for x in (ret, evi, match, sim)]
    kd, vd = (rep(x).to(F.torch_dtype(dtype)) for x in (k, v))
    for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
        refs = merge_reference(O.OracleParams(1, 1, 1, D, L, 1, B, merge_mode=mode), k, v, ret, evi, match, sim.astype(np.float64), dtype)
        fp = gpu_params(O.OracleParams(1, heads, heads, D, L, 1, B, merge_mode=mode), dtype)
        ws = F.alloc_workspace(fp)
        out = [torch.full((1, heads, B, D + 8), float("nan"), dtype=F.torch_dtype(dtype), device="cuda")[..., :D] for _ in range(2)]
        F.flowmm_merge(fp, kd, vd, *lists, out[0], out[1], ws)
        assert F.flowmm_last_device_status(ws) == 0
        for got, (ref, bound) in zip(out, refs):
            assert np.all(np.abs(got[:, :1].double().cpu().numpy() - ref) <= bound), mode
            assert torch.equal(got, got[:, :1].expand(-1, heads, -1, -1))


def test_many_rows_draw_their_windows():
    """1.6 million rows of 160 heads: windows of 64 from the counter."""
    rng = np.random.default_rng(3)
    heads, B, D = 160, 1000, 64
    n = _members("edges_apart", B, rng)
    n[300:340] = rng.integers(100, 160, 40)
    E = int(n.sum())
    L = E + B
    assert heads * L >= 1300000
    k, v = (small_integers(rng, (1, 1, L, D)) for _ in range(2))
    ret = np.sort(rng.choice(L, B, replace=False))
    evi = np.setdiff1d(np.arange(L), ret)
    match = rng.permutation(np.repeat(np.arange(B), n))
    ret, evi, match = (x.astype(np.int32)[None, None] for x in (ret, evi, match))
    sim = rng.random((1, 1, E)).astype(np.float32)
    refs = merge_reference(O.OracleParams(1, 1, 1, D, L, 1, B, merge_mode=F.MERGE_MEAN), k, v, ret, evi, match, sim.astype(np.float64), F.BF16)
    rep = lambda x: torch.from_numpy(np.ascontiguousarray(np.repeat(x, heads, 1))).cuda()
    fp = gpu_params(O.OracleParams(1, heads, heads, D, L, 1, B, merge_mode=F.MERGE_MEAN), F.BF16)
    out = [torch.full((1, heads, B, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    F.flowmm_merge(fp, rep(k).bfloat16(), rep(v).bfloat16(), *(rep(x) for x in (ret, evi, match, sim)), out[0], out[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    for got, (ref, bound) in zip(out, refs):
        assert np.all(np.abs(got[:, :1].double().cpu().numpy() - ref) <= bound)
        assert torch.equal(got, got[:, :1].expand(-1, heads, -1, -1))


@pytest.mark.parametrize("E", [1, 33, 300, 2047, 2048, 2049, 4096])
def test_lists_of_many_heads(E):
    """150 heads, so a block per head: positions kept from the first walk (up to 2048) and staged, a sixth of them dropped."""
    rng = np.random.default_rng(E)
    heads, B, D = 150, 700, 128
    L = E + B
    k, v = (small_integers(rng, (1, 1, L, D)) for _ in range(2))
    ret = np.sort(rng.choice(L, B, replace=False))
    evi = np.setdiff1d(np.arange(L), ret)
    match = np.where(rng.random(E) < 1 / 6, -1, np.minimum(rng.integers(0, B, E), rng.integers(0, 2 * B, E)))   # (some slots popular)
    sim = np.where(match >= 0, rng.random(E), 0).astype(np.float32)[None, None]
    ret, evi, match = (x.astype(np.int32)[None, None] for x in (ret, evi, match))
    rep = lambda x: torch.from_numpy(np.ascontiguousarray(np.repeat(x, heads, 1))).cuda()
    lists = [rep(x) for x in (ret, evi, match, sim)]
    for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
        refs = merge_reference(O.OracleParams(1, 1, 1, D, L, 1, B, merge_mode=mode), k, v, ret, evi, match, sim.astype(np.float64), F.BF16)
        fp = gpu_params(O.OracleParams(1, heads, heads, D, L, 1, B, merge_mode=mode), F.BF16)
        out = [torch.full((1, heads, B, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        ws = F.alloc_workspace(fp)
        F.flowmm_merge(fp, rep(k).bfloat16(), rep(v).bfloat16(), *lists, out[0], out[1], ws)
        assert F.flowmm_last_device_status(ws) == 0
        for got, (ref, bound) in zip(out, refs):
            assert np.all(np.abs(got[:, :1].double().cpu().numpy() - ref) <= bound), mode
            assert torch.equal(got, got[:, :1].expand(-1, heads, -1, -1))


@pytest.mark.parametrize("dtype,D,E", [(F.BF16, 128, 0), (F.BF16, 64, 0), (F.BF16, 64, 1), (F.F32, 64, 0), (F.F32, 128, 1)])
def test_rows_gigabytes_apart(dtype, D, E):
    """Two or three rows, 4 GiB between one and the next (a byte offset that 32 bits do not hold): pivots alone, and a merged row of
    each of so many heads, all on the same rows, that their lists are sorted."""
    B, heads = 2, 1 if E == 0 else 20000
    L, apart = B + E, 2 ** 32 // torch.empty((), dtype=F.torch_dtype(dtype)).element_size()
    rows = torch.arange(1, 1 + L * D, device="cuda").reshape(L, D).remainder(50).to(F.torch_dtype(dtype))
    k, v = (torch.zeros((L - 1) * apart + D, dtype=F.torch_dtype(dtype), device="cuda").as_strided((1, heads, L, D), (0, 0, apart, 1)) for _ in range(2))
    k[0, 0], v[0, 0] = rows, rows.flip(0)
    fp = F.Params(1, heads, heads, D, L, 1, B, dtype=dtype, merge_mode=F.MERGE_MEAN)
    ret = torch.tensor([0, L - 1], dtype=torch.int32, device="cuda").expand(1, heads, B).contiguous()
    evi, match = (torch.full((1, heads, E), x, dtype=torch.int32, device="cuda") for x in (1, 0))
    out = [torch.full((1, heads, B, D), float("nan"), dtype=F.torch_dtype(dtype), device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    F.flowmm_merge(fp, k, v, ret, evi, match, torch.zeros((1, heads, E), device="cuda"), out[0], out[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    for got, src in zip(out, (rows, rows.flip(0))):
        want = src[[0, L - 1]].clone()
        if E:
            want[0] = ((src[0].float() + src[1].float()) / 2).to(want.dtype)     # (exact: halves of small integers)
        assert torch.equal(got, want.expand(1, heads, B, D))


@pytest.mark.parametrize("n", [100, 128])
def test_many_rows_sum_long_slots_in_parts_of_64(n):
    """1.3 million rows, whose windows are drawn from the counter: a slot's first 64 members add up to 2^24, the others are ones, which
    vanish if they are added to that one by one.  With the parts added up on their own only the last sum and the mean round:
    2^-22 relative covers both; all ones lost would be 64 / 2^24."""
    heads, B, D = 160, 300, 64
    E = 30 * n
    L = E + B
    heads = -(-1310000 // L)
    ret = np.arange(B)                                              # (every tenth slot is long, the others have no members)
    evi = np.arange(B, L)
    match = np.repeat(np.arange(0, B, 10), n)
    k = np.ones((L, D), np.float32)
    k[B:][np.arange(E) % n < 64] = 2.0 ** 18
    k *= np.arange(1, D + 1) % 3 + 1
    kd = torch.from_numpy(k).cuda().expand(1, heads, L, D)
    rep = lambda x, t: torch.from_numpy(np.ascontiguousarray(np.broadcast_to(x.astype(t), (1, heads, x.size)))).cuda()
    fp = F.Params(1, heads, heads, D, L, 1, B, dtype=F.F32, merge_mode=F.MERGE_MEAN)
    ws = F.alloc_workspace(fp)
    out = [torch.full((1, heads, B, D), float("nan"), device="cuda") for _ in range(2)]
    F.flowmm_merge(fp, kd, kd, rep(ret, np.int32), rep(evi, np.int32), rep(match, np.int32), rep(np.zeros(E), np.float32), out[0], out[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    k64 = k.astype(np.float64)
    want = k64[:B].copy()
    want[::10] = (k64[:B:10] + k64[B:].reshape(30, n, D).sum(1)) / (n + 1)
    for got in out:
        assert torch.equal(got, got[:, :1].expand(-1, heads, -1, -1))
        assert np.abs(got[0, 0].double().cpu().numpy() / want - 1).max() < 2.0 ** -22
