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


@pytest.mark.parametrize("D,dtype", [(128, F.BF16), (64, F.BF16), (128, F.F32)])
def test_decode_workspace_never_shrinks_and_stays_small(lib, D, dtype):
    """More keys or heads never ask for less; a head is given room for eight records, or as many as its ranges of 1920 keys, only
    while four ranges per SM of a B200 come to that many."""
    def size(uh, keys, G):
        n, cp = ctypes.c_size_t(0), F._CDecodeParams(uh, G, 1, D, keys, dtype, 0.0, F.PATH_AUTO)
        assert lib.flowmm_decode_workspace_bytes(ctypes.byref(cp), ctypes.byref(n)) == 0
        return n.value
    for uh in (1, 4, 33, 74, 75, 296, 591, 592, 2560):
        sizes = [size(uh, keys, 4) for keys in sorted(set(range(1, 40000, 61)) | set(range(37880, 37900)) | set(range(15300, 15400)))]
        assert sizes == sorted(sizes), uh
    for keys in (1, 128, 129, 1690, 15361, 33792):
        sizes = [size(uh, keys, 4) for uh in range(1, 1300)]
        assert sizes == sorted(sizes), keys
    for uh, keys, G in ((2560, 1690, 8), (296, 1690, 8), (8, 33792, 8), (1, 100, 1)):
        ranges = -(-keys // 1920)
        assert size(uh, keys, G) <= 512 + max(uh * ranges, 592 + (min(uh, 74) if (D, dtype) == (128, F.BF16) else uh)) * G * (D + 2) * 4
