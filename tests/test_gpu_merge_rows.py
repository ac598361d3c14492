"""Merge of sorted lists by windows of rows: slots of chosen numbers of members (none, the most that stay whole, one more, several
pieces) at chosen places of a window, windows of 16 to 32 and of 64 rows, taken with a stride or drawn from the counter,
pieces of long slots as items of their own and spread over the windows, every row width, heads and units that differ, and layouts of
all tensors with gaps or other strides.
The values let one lost or doubled member be seen (test_merge_reference.py)."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F

from gpu_util import gpu_params, merge_reference, small_integers

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


def _window(heads, L, B):
    """Rows of a window, and whether the pieces of long slots are items of their own, by the library's rule: the shortest windows by which
    each of 3552 warps has one at most and some are left for pieces."""
    if heads * L >= 1300000:
        return 64, False
    win = 16 if heads * L < 40000 else next(w for w in range(16, 36, 4) if w == 32 or (
        w * B >= 2 * L and heads * (-(-L // w) + (L - B) // 256) <= 3552))
    return win, heads * (-(-L // win) + 2 * ((L - B) // 64) + 2) <= 2 * 3552


def _lists(rng, B, E, counts):
    """Pivots, non-pivots and matches of heads whose slots have these numbers of members, [variants, .]; what is left of E is dropped."""
    L = B + E
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in counts])
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret])
    match = np.stack([rng.permutation(np.concatenate([np.repeat(np.arange(B), n), np.full(E - n.sum(), -1)])) for n in counts])
    sim = np.where(match >= 0, rng.random(match.shape), 0)
    return ret.astype(np.int32), evi.astype(np.int32), match.astype(np.int32), sim.astype(np.float32)


def _heads(x, U, H, roll=False):
    """[variants, ...] as [U, H, ...] on the GPU: the heads have the variants by turns, their rows' columns rolled by the head's number,
    so that a row or a list of another head shows."""
    x = torch.from_numpy(x).cuda()
    return torch.stack([x[i % len(x)].roll(i, -1) if roll else x[i % len(x)] for i in range(U * H)]).reshape(U, H, *x.shape[1:])


def _gaps(x):
    """The same values with NaN between rows, heads and units (gaps of 16 bytes' multiples)."""
    U, H, L, D = x.shape
    row, head = D + 8, L * (D + 8) + 24
    return torch.full((U * H * head + U * 8,), float("nan"), device="cuda", dtype=x.dtype).as_strided((U, H, L, D), (H * head + 8, head, row, 1)).copy_(x)


def _check_merge(rng, U, H, B, E, D, dtype, mode, counts):
    """K by tokens first, V and the outputs with gaps, against the oracle for each of the variants."""
    L = B + E
    k, v = (small_integers(rng, (1, len(counts), L, D)) for _ in range(2))
    lists = _lists(rng, B, E, counts)
    ref_p = O.OracleParams(1, len(counts), len(counts), D, L, 1, B, merge_mode=mode)
    refs = merge_reference(ref_p, k, v, *(x[None] for x in lists[:3]), lists[3][None].astype(np.float64), dtype)
    kd, vd = (_heads(x[0], U, H, roll=True).to(F.torch_dtype(dtype)) for x in (k, v))
    kd = kd.transpose(1, 2).contiguous().transpose(1, 2)
    fp = gpu_params(O.OracleParams(U, H, H, D, L, 1, B, merge_mode=mode), dtype)
    ws = F.alloc_workspace(fp)
    out = [torch.full((U, H, B, D + 8), float("nan"), dtype=F.torch_dtype(dtype), device="cuda")[..., :D] for _ in range(2)]
    F.flowmm_merge(fp, kd, _gaps(vd), *(_heads(x, U, H) for x in lists), out[0], out[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    for got, (ref, bound) in zip(out, refs):
        assert torch.all((got.double() - _heads(ref[0], U, H, roll=True)).abs() <= _heads(bound[0], U, H, roll=True))


@pytest.mark.parametrize("dtype,D", [(F.BF16, 128), (F.BF16, 64), (F.F32, 64), (F.F32, 128)])
@pytest.mark.parametrize("U,H", [(1, 1), (4, 5), (5, 5), (2, 45)])  # windows of 16, of 28 and of 32 with pieces of their own, of 32 with pieces spread
@pytest.mark.parametrize("pattern", ["edges_first", "edges_apart", "edges_last", "alternate"])
def test_slots_of_chosen_sizes(pattern, U, H, dtype, D):
    rng = np.random.default_rng(D + U * H)
    B = 700
    counts = [_members(pattern, B, rng) for _ in range(min(U * H, 7))]
    E = max(int(n.sum()) for n in counts) + 150
    assert E > 1024                                                 # (no short list)
    few = pattern == "alternate"
    assert _window(U * H, E + B, B) == {1: (16, True), 20: (16 if few else 28, True), 25: (20 if few else 32, True), 90: (32, False)}[U * H]
    for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
        _check_merge(rng, U, H, B, E, D, dtype, mode, counts)


@pytest.mark.parametrize("H,B,win", [(16, 700, 20), (20, 700, 28), (23, 700, 32), (16, 2000, 20), (20, 2000, 24), (23, 2000, 28), (12, 250, 32)])
@pytest.mark.parametrize("dtype,D", [(F.BF16, 128), (F.F32, 64)])
def test_windows_in_between(H, B, win, dtype, D):
    """Windows of 20, 24 and 28 rows; and few slots, where windows are not shorter than two of them."""
    rng = np.random.default_rng(H + D)
    counts = [_members(p, B, rng) for p in (("edges_apart", "edges_last", "alternate") if B < 2000 else ("alternate",))]
    E = 4000 - B
    assert _window(H, 4000, B) == (win, True) and max(n.sum() for n in counts) < E
    _check_merge(rng, 1, H, B, E, D, dtype, F.MERGE_EXPSIM, counts)


def test_many_rows_draw_their_windows():
    """1.6 million rows of 160 heads: windows of 64 from the counter."""
    rng = np.random.default_rng(3)
    B = 1000
    counts = [_members("edges_apart", B, rng) for _ in range(7)]
    for n in counts:
        n[300:340] = rng.integers(100, 160, 40)
    E = max(int(n.sum()) for n in counts)
    assert 160 * (E + B) >= 1300000
    _check_merge(rng, 2, 80, B, E, 64, F.BF16, F.MERGE_MEAN, counts)


@pytest.mark.parametrize("E", [1, 33, 300, 2047, 2048, 2049, 4096])
def test_lists_of_many_heads(E):
    """150 heads, so a block per head: positions kept from the first walk (up to 2048) and staged, about a sixth of them dropped."""
    rng = np.random.default_rng(E)
    B = 700
    counts = []
    for _ in range(7):                                              # (some slots popular)
        match = np.where(rng.random(E) < 1 / 6, -1, np.minimum(rng.integers(0, B, E), rng.integers(0, 2 * B, E)))
        counts.append(np.bincount(match[match >= 0], minlength=B))
    for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
        _check_merge(rng, 2, 75, B, E, 128, F.BF16, mode, counts)


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
