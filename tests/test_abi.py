"""The C-ABI library builds, loads without a GPU and exports every symbol the header declares;
host-only validation works without any CUDA call."""
import ctypes
import os
import re

import pytest

from paper_2511_05534_b200 import binding as F
from paper_2511_05534_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return F.load()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "flowmm.h")).read()
    declared = set(re.findall(r"\b(flowmm_[a-z_]+)\s*\(", header))
    assert declared, "no declarations found"
    for name in declared:
        assert hasattr(lib, name), name
    assert declared == set(F.EXPORTS)


def test_params_struct_matches_header():
    header = open(os.path.join(ROOT, "include", "flowmm.h")).read()
    body = header[header.index("typedef struct {"):header.index("} flowmm_params;")]
    fields = re.findall(r"(?:int32_t|float|int64_t)\s+([^;]+);", body)
    names = [n.strip().split("[")[0] for group in fields for n in group.split(",")]
    assert names == [f[0] for f in F._CParams._fields_]


def test_workspace_bytes_and_validation_need_no_gpu(lib):
    p = F.Params(4, 8, 2, 128, 1000, 16, 100)
    n = F.flowmm_workspace_bytes(p)
    assert n > 0 and n % 256 == 0
    bigger = F.flowmm_workspace_bytes(F.Params(8, 8, 2, 128, 1000, 16, 100))
    assert bigger > n
    cases = [
        (dict(n_q_heads=7), 2), (dict(head_dim=96), 2), (dict(window=2000), 2), (dict(n_keep=0), 3),
        (dict(n_keep=1001), 3), (dict(keep_window=1, n_keep=8), 3), (dict(dtype=5), 4), (dict(n_units=0), 2),
    ]
    for change, code in cases:
        kw = dict(n_units=4, n_q_heads=8, n_kv_heads=2, head_dim=128, seq_len=1000, window=16, n_keep=100)
        kw.update(change)
        with pytest.raises(F.FlowmmError) as e:
            F.flowmm_workspace_bytes(F.Params(**kw))
        assert e.value.code == code, change
    assert F.status_string(0) == "ok" and "workspace" in F.status_string(5)


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(F, "_lib", None)
    monkeypatch.setattr(F, "LIB_PATH", str(tmp_path / "libflowmm.so"))
    with pytest.raises(FileNotFoundError):
        F.load()


@pytest.mark.parametrize("Hkv,G,W,D,dtype", [(4, 7, 32, 128, F.BF16), (8, 8, 64, 128, F.BF16), (32, 1, 32, 128, F.BF16), (1, 8, 128, 128, F.BF16),
                                             (3, 5, 32, 128, F.BF16), (4, 4, 16, 64, F.F32), (1, 4, 100, 128, F.F32)])
def test_workspace_never_shrinks_with_the_problem(lib, Hkv, G, W, D, dtype):
    """A workspace kept for the most units and the longest context serves the smaller calls of the same budget, across the lines at which
    windows, chunks and items change size."""
    size = lambda U, L, B: F.flowmm_workspace_bytes(F.Params(U, G * Hkv, Hkv, D, L, W, B, dtype=dtype))
    for U in (1, 2, 5, 28):
        for B in (16, 500):
            lengths = sorted({max(B, W) + i for i in range(900)} | set(range(max(B, W), 45000, 37)) | {40000 // (U * Hkv) + i for i in range(-300, 300)} |
                             {1300000 // (U * Hkv) + i for i in range(-300, 300)})
            sizes = [size(U, L, B) for L in lengths if L >= max(B, W)]
            assert sizes == sorted(sizes), (U, B)
    for L, B in ((200, 50), (640, 64), (2176, 217), (33792, 1690)):
        sizes = [size(U, L, B) for U in range(1, 320)]
        assert sizes == sorted(sizes), (L, B)
