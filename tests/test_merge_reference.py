"""The bounds that the GPU tests of the merge lists use accept the right result and reject one with a single member lost, doubled or
in another slot, at the longest lists of those tests.  The mistakes are made in the oracle's inputs; nothing here needs a GPU."""
import numpy as np
import pytest

from oracle import compare, flowmm_oracle as O
from paper_2511_05534_b200 import binding as F

from gpu_util import merge_reference, small_integers


@pytest.mark.parametrize("dtype", [F.F32, F.BF16])
@pytest.mark.parametrize("E,B,kind", [(33000, 257, "one"), (33000, 257, "spread"), (70000, 300, "one"), (70000, 300, "spread"), (1024, 300, "one")])
def test_one_wrong_member_is_seen(E, B, kind, dtype):
    rng = np.random.default_rng(E)
    L, D = E + B, 128
    p = O.OracleParams(1, 1, 1, D, L, 1, B, merge_mode=F.MERGE_MEAN)
    k, v = (small_integers(rng, (1, 1, L, D)) for _ in range(2))
    ret = np.sort(rng.choice(L, B, replace=False))[None, None].astype(np.int32)
    evi = np.setdiff1d(np.arange(L), ret[0, 0])[None, None].astype(np.int32)
    match = rng.integers(0, B, (1, 1, E)).astype(np.int32) if kind == "spread" else np.full((1, 1, E), B - 1, dtype=np.int32)
    sim = np.zeros((1, 1, E))
    refs = merge_reference(p, k, v, ret, evi, match, sim, dtype)
    rounded = compare.round_bf16 if dtype == F.BF16 else (lambda x: x.astype(np.float32).astype(np.float64))
    fits = lambda outs: all(np.all(np.abs(rounded(o) - ref) <= bound) for o, (ref, bound) in zip(outs, refs))
    assert fits([r for r, _ in refs])
    for j in rng.choice(E, 5, replace=False):
        for wrong in (-1, int(match[0, 0, j] + 1) % B):            # lost; in the next slot
            m = match.copy()
            m[0, 0, j] = wrong
            assert not fits(O.merge(p, k, v, ret, evi, m, sim)[:2])
        i = int(np.flatnonzero(match[0, 0] == match[0, 0, j])[0]) # doubled, in another member's place
        e = evi.copy()
        e[0, 0, i if i != j else np.flatnonzero(match[0, 0] == match[0, 0, j])[1]] = evi[0, 0, j]
        assert not fits(O.merge(p, k, v, ret, e, match, sim)[:2])
