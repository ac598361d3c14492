"""Exponentials of the scoring and flow epilogues where they are exp2 of the hardware in every column: chunks of 32 keys under the
causal mask or of both modalities, proxy rows of both modalities.  Logits are chosen so that one key's, or one row's, exponential is
the whole of a result's error, over the residues of its position and over the fractions that exp2 sees.

Tolerance: exp2.approx is within 2^-22 of its value, its argument (below 2 in magnitude, a product of two rounded factors) within
2^-22, which is 1.7e-7 of the value; sums of at most 64 equal terms in at least four chains, the normaliser's logarithm and the
quotient round at 2^-24 a dozen times at most: 1.2e-6 together.  A polynomial with an error of 3.6e-6 in some columns does not pass."""
import numpy as np
import pytest
import torch

from oracle import flowmm_oracle as O
from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import inputs

from gpu_util import gpu_params, to_dev

pytestmark = pytest.mark.gpu
D, ROOT = 128, 128.0 ** 0.5
C = np.linspace(0.35, 1.04, 64)                                      # minus the logit: its exp2 argument runs over [-1.5, -0.5]


def _bf16(x):
    return inputs.round_to_bf16(np.ascontiguousarray(x, dtype=np.float32))


def _score(p, q, k, m):
    imp, cross, _ = O.score(p, q, k, m)
    g_imp, g_cross = torch.full(imp.shape, float("nan"), device="cuda"), torch.full(cross.shape, float("nan"), device="cuda")
    ws = F.alloc_workspace(gpu_params(p, F.BF16))
    F.flowmm_score(gpu_params(p, F.BF16), to_dev(q, F.BF16), to_dev(k, F.BF16), torch.from_numpy(m).cuda(), g_imp, g_cross, ws)
    assert F.flowmm_last_device_status(ws) == 0
    return imp, cross, g_imp.double().cpu().numpy(), g_cross.double().cpu().numpy()


@pytest.mark.parametrize("L", [32, 64])
def test_flow_of_one_visual_token(L):
    """Rows after the one visual token see it in the chunk on the diagonal (L = 32), or in an earlier one of both modalities as well.  Its
    own row is all but blind to the text."""
    U, H = 8, len(C)
    q, k = np.zeros((U, H, L, D)), np.zeros((U, H, L, D))
    m = np.zeros((U, L), np.uint8)
    q[..., 0] = C[:, None] * ROOT
    k[:, :, 1:, 0] = -1
    for u in range(U):
        q[u, :, 8 + u, 0], q[u, :, 8 + u, 1], k[u, :, 8 + u, 1], m[u, 8 + u] = 0, 40 * ROOT, 1, 1
    q, k = _bf16(q), _bf16(k)
    cross = O.score(O.OracleParams(U, H, H, D, L, L, 1), q, k, m)[1]
    fp = F.Params(U, H, H, D, L, 1, 1)
    g_cross, rho, strat = torch.zeros((U, H), device="cuda"), torch.zeros(U, device="cuda"), torch.zeros(U, dtype=torch.int32, device="cuda")
    ws = torch.zeros(F.flowmm_full_flow_workspace_bytes(fp), dtype=torch.uint8, device="cuda")
    F.flowmm_full_flow(fp, to_dev(q, F.BF16), to_dev(k, F.BF16), torch.from_numpy(m).cuda(), g_cross, rho, strat, ws)
    assert F.flowmm_last_device_status(ws) == 0
    assert np.abs(g_cross.double().cpu().numpy() / cross - 1).max() < 1.2e-6


@pytest.mark.parametrize("H,G", [(32, 2), (7, 3)])                   # two passes; few heads: one pass by clusters
def test_normalisers_of_masked_chunks(H, G):
    """All of a proxy row's mass is on the first key and on the window's keys of one residue (mod 8)."""
    U, W, L = 8, 32, 320
    q, k = np.zeros((U, G * H, W, D)), np.zeros((U, H, L, D))
    q[..., 0], q[..., 1] = C[:G * H, None] * ROOT, ROOT
    k[:, :, 1:, 1] = -60
    for u in range(U):
        k[u, :, L - W + u::8, 0], k[u, :, L - W + u::8, 1] = -1, 0
    imp, _, g_imp, _ = _score(O.OracleParams(U, G * H, H, D, L, W, 1), _bf16(q), _bf16(k), np.zeros((U, L), np.uint8))
    on = imp > 1e-3
    assert on.sum() == U * H * 5 and np.abs(g_imp[on] / imp[on] - 1).max() < 1.2e-6


@pytest.mark.parametrize("W,H,G", [(32, 32, 2), (64, 32, 2), (128, 32, 2), (32, 7, 3), (64, 7, 2), (128, 7, 1)])
def test_importances_from_a_window_of_both_modalities(W, H, G):
    """Keys that the window's rows of one residue (mod 8) alone see; every word of 32 rows has both modalities."""
    U, L = 8, 512
    q, k = np.zeros((U, G * H, W, D)), np.zeros((U, H, L, D))
    q[..., 1] = ROOT
    q[..., 2] = ROOT
    for u in range(U):
        q[u, :, u::8, 0], q[u, :, u::8, 2] = C[:G * H, None] * ROOT, 0
    k[:, :, 1:, 1] = -60
    k[:, :, 8:128:8, 0], k[:, :, 8:128:8, 1], k[:, :, 8:128:8, 2] = -1, 0, -60
    m = np.ascontiguousarray(np.broadcast_to(np.arange(L) // 16 % 2, (U, L)), dtype=np.uint8)
    imp, _, g_imp, _ = _score(O.OracleParams(U, G * H, H, D, L, W, 1), _bf16(q), _bf16(k), m)
    assert np.abs(g_imp[:, :, 8:128:8] / imp[:, :, 8:128:8] - 1).max() < 1.2e-6


@pytest.mark.parametrize("W,G", [(32, 2), (32, 3), (32, 4), (64, 1), (64, 2), (64, 3)])
@pytest.mark.parametrize("H", [7, 32])                               # one pass by clusters; two passes
def test_importances_in_front_of_the_window(W, G, H):
    """Keys in front of the window in its tile of 128: one per chunk of 32, of residue u (mod 8), that all proxy rows see with one logit, against
    one that has the chunk's maximum."""
    U, L = 8, 256
    q, k = np.zeros((U, H * G, W, D)), np.zeros((U, H, L, D))
    q[..., 0], q[..., 1] = np.repeat(np.resize(C, U * H).reshape(U, H), G, 1)[:, :, None] * ROOT, ROOT
    k[:, :, 1:, 1] = -60
    for u in range(U):
        k[u, :, 144 + u:L - W:32, 0] = -1
        for first in (144 + u, 128 + (u + 4) % 8):
            k[u, :, first:L - W:32, 1] = 0
    imp, _, g_imp, _ = _score(O.OracleParams(U, H * G, H, D, L, W, 1), _bf16(q), _bf16(k), np.zeros((U, L), np.uint8))
    for u in range(U):
        ref, got = (x[u, :, 144 + u:L - W:32] / x[u, :, 128 + (u + 4) % 8:L - W:32] for x in (imp, g_imp))
        assert ref.min() > 0.3 and np.abs(got / ref - 1).max() < 1.2e-6


@pytest.mark.parametrize("few", [0, 1])
@pytest.mark.parametrize("logit", [-10, -14, -17, -25, -60])
def test_small_masses_in_chunks_of_both_modalities(few, logit):
    """Chunks in which one modality has a share of 1e-4 to 1e-26, and a window of the other one, whose cross-modal mass it is.  Tolerance: the
    polynomial's 3.6e-6 in numerator and normaliser, and the exp2 argument, which is as large as 87 (1e-5 of the value)."""
    U, H, W, L = 2, 4, 32, 513
    rng = np.random.default_rng(1)
    m = (rng.random((U, L)) < 0.5).astype(np.uint8)
    m[:, L - W:] = 1 - few
    q, k = np.zeros((U, 2 * H, W, D)), 0.25 * rng.standard_normal((U, H, L, D))
    q[..., 0] = ROOT
    k[..., 0] = np.where(m == few, logit, 0)[:, None]
    _, cross, _, g_cross = _score(O.OracleParams(U, 2 * H, H, D, L, W, 1), _bf16(q), _bf16(k), m)
    assert np.abs(g_cross / cross - 1).max() < 2e-5
