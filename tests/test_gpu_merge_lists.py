"""Member lists of the gather merge at the edges of their builders: a CTA or a cluster of two, four or eight per head (2048,
4096, 8192 non-pivots), the counting sort for many heads (short and long lists), odd and even slot counts, budgets too large for the
clusters (5459 pivots) and those of which an SM holds one CTA (2729), lists that leave shared memory (70 000 non-pivots),
everything dropped, everything in one slot.  The step
is called on its own with hand-made matches, on values that let one lost or doubled member be seen (test_merge_reference.py)."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F

from gpu_util import gpu_params, merge_reference, small_integers, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,B,heads", [(1, 241, 2), (31, 242, 2), (2047, 250, 2), (2048, 251, 2), (4096, 241, 2), (8191, 300, 2), (8192, 301, 2),
                                       (9000, 1691, 2), (20000, 2501, 2), (33000, 257, 2), (9000, 2800, 2), (4096, 241, 300), (4097, 300, 300),
                                       (9000, 2800, 16), (9000, 5459, 2), (9000, 5460, 2), (70000, 300, 1), (38500, 300, 2)])
@pytest.mark.parametrize("kind", ["spread", "dropped", "one"])
def test_merge_of_hand_made_matches(E, B, heads, kind):
    rng = np.random.default_rng(E + B)
    U, Hkv, D, L = 1, heads, 128, E + B
    n = min(Hkv, 2)                                                 # (many heads repeat the data of two)
    rep = lambda x: np.ascontiguousarray(np.tile(x, (1, Hkv // n) + (1,) * (x.ndim - 2)))
    k, v = (small_integers(rng, (U, n, L, D)) for _ in range(2))
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in range(n)])[None].astype(np.int32)
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32)
    match = rng.integers(-1, B, (U, n, E)).astype(np.int32)
    if kind == "dropped":
        match[rng.random((U, n, E)) < 0.9] = -1
        match[0, -1] = -1
    elif kind == "one":
        match[:] = B - 1
    sim = np.where(match >= 0, rng.random((U, n, E)), 0).astype(np.float32)
    t = lambda x: torch.from_numpy(rep(x)).cuda()
    lists = [t(x) for x in (ret, evi, match, sim)]
    for dtype in (F.BF16, F.F32):                                   # (both take the same lists; fp32 shows every member)
        kd, vd = (t(x).to(F.torch_dtype(dtype)) for x in (k, v))
        for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
            refs = merge_reference(O.OracleParams(U, n, n, D, L, 1, B, merge_mode=mode), k, v, ret, evi, match, sim.astype(np.float64), dtype)
            fp = gpu_params(O.OracleParams(U, Hkv, Hkv, D, L, 1, B, merge_mode=mode), dtype)
            g = [torch.full((U, Hkv, B, D), float("nan"), dtype=F.torch_dtype(dtype), device="cuda") for _ in range(2)]
            ws = F.alloc_workspace(fp)
            F.flowmm_merge(fp, kd, vd, *lists, g[0], g[1], ws)
            assert F.flowmm_last_device_status(ws) == 0
            for got, (ref, bound) in zip(g, refs):                  # the last heads are compared, and the others with them
                assert np.all(np.abs(got[:, Hkv - n:].double().cpu().numpy() - ref) <= bound), (dtype, mode)
                assert torch.equal(got.view(U, Hkv // n, n, B, D), got[:, Hkv - n:].unsqueeze(1).expand(-1, Hkv // n, -1, -1, -1))


@pytest.mark.parametrize("dtype,D", [(F.F32, 64), (F.F32, 128), (F.BF16, 64), (F.BF16, 128)])
@pytest.mark.parametrize("E,B,heads", [(1, 300, 1), (32, 257, 2), (33, 249, 40), (1023, 248, 1), (1024, 300, 30), (1025, 300, 2)])
@pytest.mark.parametrize("kind", ["spread", "popular"])
def test_short_lists(dtype, D, E, B, heads, kind):
    """Lists up to 1024 non-pivots are merged straight from the matches: one slot or four per warp, slots of up to 64 members and
    of more, rows of one to two 16-byte vectors per lane."""
    rng = np.random.default_rng(E + B + D)
    L = E + B
    k, v = (small_integers(rng, (1, heads, L, D)) for _ in range(2))
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in range(heads)])[None].astype(np.int32)
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32)
    match = rng.integers(-1, B, (1, heads, E)).astype(np.int32)
    if kind == "popular":                                           # a few slots of 64, 65 and many members
        match[..., : E // 2] = 7
        match[..., E // 2: E // 2 + 65] = B - 1
        match[..., E // 2 + 65: E // 2 + 129] = 0
    sim = np.where(match >= 0, rng.random((1, heads, E)), 0).astype(np.float32)
    t = lambda x: torch.from_numpy(x).cuda()
    for mode in (F.MERGE_MEAN, F.MERGE_EXPSIM):
        p = O.OracleParams(1, heads, heads, D, L, 1, B, merge_mode=mode)
        g = [torch.full((1, heads, B, D), float("nan"), dtype=F.torch_dtype(dtype), device="cuda") for _ in range(2)]
        fp = gpu_params(p, dtype)
        ws = F.alloc_workspace(fp)
        F.flowmm_merge(fp, to_dev(k, dtype), to_dev(v, dtype), t(ret), t(evi), t(match), t(sim), g[0], g[1], ws)
        assert F.flowmm_last_device_status(ws) == 0
        for got, (ref, bound) in zip(g, merge_reference(p, k, v, ret, evi, match, sim.astype(np.float64), dtype)):
            assert np.all(np.abs(got.double().cpu().numpy() - ref) <= bound), mode


@pytest.mark.parametrize("B", [65535 * 32, 65535 * 32 + 1])
def test_short_list_with_more_slots_than_a_grid_has_rows(B):
    """256 non-pivots and budgets around two million: the last one that a grid of short-list blocks covers and the first that
    goes to the persistent kernels.  Pivots without members come back bit for bit; the others as the sum says."""
    E, D, H = 256, 64, 1
    L = E + B
    gen = torch.Generator(device="cuda").manual_seed(B)
    k, v = (torch.randn((1, H, L, D), device="cuda", generator=gen).bfloat16() for _ in range(2))
    rng = np.random.default_rng(1)
    evi = torch.from_numpy(np.sort(rng.choice(L, E, replace=False))).cuda()
    keep = torch.ones(L, dtype=torch.bool, device="cuda")
    keep[evi] = False
    ret = keep.nonzero()[:, 0]
    match = torch.from_numpy(rng.integers(0, B, E)).cuda()
    match[0], match[1:70], match[70] = -1, B - 1, 0
    sim = torch.rand(E, device="cuda", generator=gen)
    p = O.OracleParams(1, H, H, D, L, 1, B)
    fp = gpu_params(p, F.BF16)
    g = [torch.zeros((1, H, B, D), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    i32 = lambda x: x.to(torch.int32).view(1, H, -1).contiguous()
    F.flowmm_merge(fp, k, v, i32(ret), i32(evi), i32(match), sim.view(1, H, E), g[0], g[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    slots = match[1:].unique()
    w = torch.exp(sim.double() - 1)[1:, None]
    for got, x in zip(g, (k, v)):
        x = x[0, 0]
        plain = torch.ones(B, dtype=torch.bool, device="cuda")
        plain[slots] = False
        assert torch.equal(got[0, 0][plain], x[ret[plain]])
        num, den = torch.zeros((B, D), dtype=torch.float64, device="cuda"), torch.ones((B, 1), dtype=torch.float64, device="cuda")
        num.index_add_(0, match[1:], w * x[evi[1:]].double())
        den.index_add_(0, match[1:], w)
        ref = ((num + x[ret].double()) / den)[slots]
        # the output's rounding to bf16 (8 bits: 2^-8 of the value), and below it fp32 sums of up to 69 members: (69 + 16) 2^-24
        # of the mean magnitude, which is below 8
        assert torch.all((got[0, 0][slots].double() - ref).abs() <= ref.abs() * 2 ** -8 + 2 ** -14)


@pytest.mark.parametrize("E,B,heads,launches", [(100, 40000, 2, 1), (256, 20000, 3, 1), (256, 2100, 32, 1), (257, 20000, 3, 2), (200, 1000, 33, 2), (200, 800, 33, 1)])
def test_few_heads_of_many_slots(E, B, heads, launches):
    """Up to 256 members of up to 32 heads go straight from the matches however many slots there are: a list builder of a block per
    head walks the slots one round after the other (2 heads of 30 000 slots took ten times as long)."""
    rng = np.random.default_rng(E + B)
    D, L = 64, E + B
    k, v = (small_integers(rng, (1, heads, L, D)) for _ in range(2))
    ret = np.sort(np.argsort(rng.random((1, heads, L)), -1)[..., :B], -1).astype(np.int32)
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32)
    match = rng.integers(-1, B, (1, heads, E)).astype(np.int32)
    sim = np.where(match >= 0, rng.random((1, heads, E)), 0).astype(np.float32)
    p = O.OracleParams(1, heads, heads, D, L, 1, B, merge_mode=F.MERGE_MEAN)
    refs = merge_reference(p, k, v, ret, evi, match, sim.astype(np.float64), F.BF16)
    fp = gpu_params(p, F.BF16)
    t = lambda x: torch.from_numpy(x).cuda()
    g = [torch.full((1, heads, B, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    F.flowmm_merge(fp, to_dev(k, F.BF16), to_dev(v, F.BF16), *(t(x) for x in (ret, evi, match, sim)), g[0], g[1], ws)
    assert F.flowmm_last_launch_count() == launches
    assert F.flowmm_last_device_status(ws) == 0
    for got, (ref, bound) in zip(g, refs):
        assert np.all(np.abs(got.double().cpu().numpy() - ref) <= bound)
