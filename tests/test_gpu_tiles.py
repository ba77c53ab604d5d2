"""GPU parity of the CUDA-core kernels at the edges of their row tiles and register units: head sizes and
feature counts that are no multiple of four, values wider than the keys, every register tile of the key
statistics, rows just below, at and above a 64-row tile, one row, and heads split over several blocks.

Tolerances are the parity gates of the other GPU tests: 1e-4 (fp32) and 2e-2 (bf16) of the oracle, floored at
the tensor's rms (outputs of the streaming form at their row's rms).
"""
import math

import pytest

import oracle
import synth
from cases import TOL, Case, relerr, relerr_rows, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


SHAPES = [
    # B, H, n, d, dv, M, L, io
    (1, 1, 1, 64, 64, 8, 8, "f32"),
    (1, 2, 63, 20, 33, 3, 5, "f32"),      # D = 15: odd, no 16-byte rows in d, dv or D
    (2, 1, 65, 34, 20, 2, 8, "bf16"),     # bf16 rows that are no multiple of 16 bytes
    (1, 3, 129, 64, 96, 8, 8, "f32"),     # 64 x 96: 4 x 4 units
    (1, 1, 130, 128, 124, 16, 8, "f32"),  # 128 x 124: 4 x 8 units, the last past the row's end
    (3, 2, 200, 48, 48, 16, 4, "bf16"),
    (1, 1, 700, 16, 128, 1, 8, "f32"),    # one projection; one head over many blocks
]


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_row_tiles(shape, causal):
    B, H, n, d, dv, M, L, io = shape
    lengths = [n] + [max(1, n // 2)] * (B - 1)
    case = Case(B, H, n, d, M, L, io, causal, seed=131, qkv_scale=1.0 / math.sqrt(d), dv=dv, lengths=lengths,
                with_grad=True)
    lu = case.luna()
    O, ref = to_host(case.run_fwd(lu)), case.oracle_fwd()
    assert (relerr_rows(O, ref) if causal else relerr(O, ref)) < TOL[io]
    for use_state in (True, False):
        g = {k: to_host(v) for k, v in case.run_bwd(lu, use_state=use_state).items()}
        rb = case.oracle_bwd()
        assert relerr(g["dV"], rb["dV"]) < TOL[io]
        if n == 1:  # one key: its weight is 1 whatever the features, so the gradients of all but V are eps-sized
            continue
        for k, which in (("dQ", "Q"), ("dK", "K")):
            ok = case.smooth_rows(which)
            assert relerr(g[k][ok], rb[k][ok]) < TOL[io], k
        for k in ("dW", "db", "dw1", "db1", "dw2", "db2"):
            assert relerr(g[k], rb[k]) < TOL[io], k


@pytest.mark.parametrize("n,d,M,L,io,causal,row0,rows", [(129, 20, 3, 5, "f32", False, 0, 129),
                                                         (65, 64, 8, 8, "bf16", True, 0, 65),
                                                         (64, 128, 16, 8, "f32", False, 63, 1),
                                                         (200, 33, 2, 8, "bf16", True, 60, 70)])
@pytest.mark.parametrize("teacher", [False, True])
def test_weight_tiles(n, d, M, L, io, causal, row0, rows, teacher):
    import torch
    import paper_2512_08061_gb300.luna as lib
    case = Case(2, 2, n, d, M, L, io, causal, seed=137, qkv_scale=1.0 / math.sqrt(d), lengths=[n, n // 2])
    lu = case.luna()
    A = torch.full((2, 2, rows, n), float("nan"), dtype=torch.float32, device="cuda")
    lib.luna_attn_weights(lu.ad, lu.pd, lu.table, case.dev["Q"], case.dev["K"], case.dev["lengths"], row0, rows,
                          teacher, A)
    ref = oracle.attn_weights(case.params, case.inp["Q"].value, case.inp["K"].value, case.lengths, causal, case.eps,
                              row0, rows, teacher)
    got = to_host(A)
    assert ((got == 0) == (ref == 0)).all()
    assert relerr(got, ref) < TOL[io]


def test_nonfinite_values_stay_in_their_column():
    """An infinite value makes its own column of the outputs non-finite and no other (both forms)."""
    import numpy as np
    import torch
    for causal in (False, True):
        case = Case(1, 1, 100, 32, 8, 8, "f32", causal, seed=139, qkv_scale=1.0 / math.sqrt(32))
        lu = case.luna()
        case.dev["V"][0, 0, 70, 5] = float("inf")
        O = to_host(case.run_fwd(lu))
        ref = case.oracle_fwd()
        rows = np.arange(100) >= (70 if causal else 0)
        assert not np.isfinite(O[0, 0, rows, 5]).any()
        keep = np.ones(O.shape, bool)
        keep[0, 0, rows, 5] = False
        assert np.isfinite(O[keep]).all()
        assert relerr(O[keep], ref[keep]) < 10 * TOL["f32"] if causal else relerr(O[keep], ref[keep]) < TOL["f32"]


@pytest.mark.parametrize("d,M", [(32, 8), (64, 8), (128, 16)])
@pytest.mark.parametrize("lengths", [False, True])
def test_many_heads_per_block(d, M, lengths):
    """bf16 forward with more heads than SMs, one or two tiles each (some sequences empty): every block changes
    heads several times, so the statistics of one head leave while the next is worked on, and the query pass's
    operand buffers are reused."""
    n = 150
    ln = [n, 0, 1, 129, 128, 77, n, 64][:8] if lengths else None
    case = Case(8, 48, n, d, M, 8, "bf16", False, seed=149, qkv_scale=1.0 / math.sqrt(d), lengths=ln)
    lu = case.luna()
    O, ref = to_host(case.run_fwd(lu)), case.oracle_fwd()
    assert relerr(O, ref) < TOL["bf16"]
    assert (to_host(case.run_fwd(lu)) == O).all()
