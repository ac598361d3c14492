"""Member lists of the gather merge at the edges of their two builders: the short and the long counting sort (4096 | 4097
non-pivots), odd and even slot counts, lists that leave shared memory (38 500 non-pivots), everything dropped, everything in
one slot.  The step is called on its own with hand-made matches."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import inputs

from gpu_util import gpu_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,B", [(1, 241), (31, 242), (4096, 241), (4097, 300), (9000, 1691), (20000, 2501), (33000, 257), (38500, 300)])
@pytest.mark.parametrize("kind", ["spread", "dropped", "one"])
def test_merge_of_hand_made_matches(E, B, kind):
    rng = np.random.default_rng(E + B)
    U, Hkv, D, L = 1, 2, 128, E + B
    p = O.OracleParams(U, Hkv, Hkv, D, L, 1, B)
    k, v = (inputs.round_to_bf16(rng.standard_normal((U, Hkv, L, D)).astype(np.float32)) for _ in range(2))
    ret = np.stack([np.sort(rng.choice(L, B, replace=False)) for _ in range(Hkv)])[None].astype(np.int32)
    evi = np.stack([np.setdiff1d(np.arange(L), r) for r in ret[0]])[None].astype(np.int32)
    match = rng.integers(-1, B, (U, Hkv, E)).astype(np.int32)
    if kind == "dropped":
        match[rng.random(match.shape) < 0.9] = -1
        match[0, 1] = -1
    elif kind == "one":
        match[:] = B - 1
    sim = np.where(match >= 0, rng.random(match.shape), 0).astype(np.float32)
    ko, vo = O.merge(p, k, v, ret, evi, match, sim.astype(np.float64))[:2]
    fp = gpu_params(p, F.BF16)
    g = [torch.zeros((U, Hkv, B, D), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = F.alloc_workspace(fp)
    t = lambda x: torch.from_numpy(x).cuda()
    F.flowmm_merge(fp, to_dev(k, F.BF16), to_dev(v, F.BF16), t(ret), t(evi), t(match), t(sim), g[0], g[1], ws)
    assert F.flowmm_last_device_status(ws) == 0
    for got, ref in zip(g, (ko, vo)):
        ref = np.asarray(ref, dtype=np.float64).reshape(U, Hkv, B, D)
        assert np.all(np.abs(got.float().cpu().numpy() - ref) <= 2e-2 + 1e-2 * np.abs(ref))
