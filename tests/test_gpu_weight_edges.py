"""GPU: attention weights at the edges of what luna_attn_weights accepts."""
import math

import numpy as np
import pytest

import oracle
from cases import TOL, Case, relerr, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


def _weights(case, lu, teacher, row0=0, rows=None):
    import torch
    import paper_2512_08061_gb300.luna as lib
    rows = case.n if rows is None else rows
    A = torch.full((case.B, case.H, rows, case.n), float("nan"), dtype=torch.float32, device="cuda")
    lib.luna_attn_weights(lu.ad, lu.pd, lu.table, case.dev["Q"], case.dev["K"], case.dev["lengths"], row0, rows,
                          teacher, A)
    return to_host(A)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("key", [0, 5, 100, 199])
def test_nan_score_reaches_its_row(key, causal):
    """A NaN key (in the first, an inner and the last tile of keys, and the first key of a thread): in every row that
    sees it the softmax has no finite sum, its own weight is NaN and every other weight 0, wherever the key lies;
    rows before it in the streaming form keep their weights."""
    n, d = 200, 32
    case = Case(1, 1, n, d, 8, 8, "f32", causal, seed=229, qkv_scale=1.0 / math.sqrt(d))
    lu = case.luna()
    ref = oracle.attn_weights(case.params, case.inp["Q"].value, case.inp["K"].value, case.lengths, causal, case.eps,
                              0, n, True)
    case.dev["K"][0, 0, key] = float("nan")
    got = _weights(case, lu, True)[0, 0]
    sees = np.arange(n) >= key if causal else np.ones(n, bool)
    assert np.isnan(got[sees, key]).all()
    assert (np.delete(got[sees], key, axis=1) == 0).all()
    if not sees.all():
        assert relerr(got[~sees], ref[0, 0][~sees]) < TOL["f32"]


@pytest.mark.parametrize("n,d,M,L,io,causal,row0,rows", [
    (1, 64, 8, 8, "f32", False, 0, 1), (4, 20, 3, 5, "f32", True, 1, 3), (31, 64, 8, 8, "bf16", True, 0, 31),
    (32, 33, 2, 8, "f32", False, 0, 32), (32, 128, 16, 8, "bf16", False, 30, 2), (33, 64, 8, 8, "f32", True, 0, 33)])
@pytest.mark.parametrize("teacher", [False, True])
def test_short_sequences(n, d, M, L, io, causal, row0, rows, teacher):
    """Sequences of one small tile: at, below and above the size where the tile changes."""
    case = Case(3, 2, n, d, M, L, io, causal, seed=233, qkv_scale=1.0 / math.sqrt(d), lengths=[n, max(1, n // 2), 1])
    ref = oracle.attn_weights(case.params, case.inp["Q"].value, case.inp["K"].value, case.lengths, causal, case.eps,
                              row0, rows, teacher)
    got = _weights(case, case.luna(), teacher, row0, rows)
    assert ((got == 0) == (ref == 0)).all()
    assert relerr(got, ref) < TOL[io]
