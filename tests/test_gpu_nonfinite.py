"""GPU: a non-finite input of the CUDA-core kernels reaches what depends on it and nothing else.

Everything else is compared with the oracle's values for the finite inputs, at the parity gate of the other tests
(1e-4, floored at the row's rms for outputs of the streaming form, at the tensor's rms otherwise).
"""
import math

import numpy as np
import pytest

from cases import TOL, Case, relerr_rows, to_host

pytestmark = pytest.mark.gpu
N, ROW, COL = 100, 70, 5  # rows 64 .. 99 are the second tile: ROW has rows before and after it in its tile


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


def _case(causal):
    case = Case(1, 1, N, 32, 8, 8, "f32", causal, seed=257, qkv_scale=1.0 / math.sqrt(32), dv=8, with_grad=True)
    return case, case.luna()


@pytest.mark.parametrize("causal", [False, True])
def test_infinite_value_in_the_outputs(causal):
    case, lu = _case(causal)
    ref = case.oracle_fwd()[0, 0]
    case.dev["V"][0, 0, ROW, COL] = float("inf")
    O = to_host(case.run_fwd(lu))[0, 0]
    sees = np.arange(N) >= (ROW if causal else 0)
    assert not np.isfinite(O[sees, COL]).any()
    keep = np.delete(np.arange(8), COL)
    assert relerr_rows(O[:, keep], ref[:, keep]) < TOL["f32"]
    if causal:
        assert relerr_rows(O[~sees], ref[~sees]) < TOL["f32"]


@pytest.mark.parametrize("which", ["V", "dO"])
@pytest.mark.parametrize("causal", [False, True])
def test_infinite_value_in_the_backward(causal, which):
    """V: the rows that see it have an infinite numerator, so their dQ and every key's dK are not finite; dV does not
    depend on V.  dO: its row's dQ, its column of dV and dK of the keys its row sees are not finite."""
    case, lu = _case(causal)
    ref = {k: case.oracle_bwd()[k][0, 0] for k in ("dQ", "dK", "dV")}
    case.run_fwd(lu)
    case.dev[which][0, 0, ROW, COL] = float("inf")
    i = np.arange(N)
    if which == "V":
        case.run_fwd(lu)
        kept = {"dQ": (i < ROW) if causal else (i < 0), "dK": i < 0, "dV": i >= 0}
        cols = np.arange(8)
    else:
        kept = {"dQ": i != ROW, "dK": (i > ROW) if causal else (i < 0), "dV": i >= 0}
        cols = np.delete(np.arange(8), COL)
    for use_state in (True, False):
        g = {k: to_host(v)[0, 0] for k, v in case.run_bwd(lu, use_state=use_state).items() if k in ref}
        for k, rows in kept.items():
            ok = rows & (np.ones(N, bool) if k == "dV" else case.smooth_rows(k[1])[0, 0])
            at = np.ix_(ok, cols if k == "dV" else np.arange(32))
            floor = np.maximum(np.abs(ref[k]), math.sqrt(np.mean(ref[k] ** 2)))
            assert np.isfinite(g[k][at]).all(), k
            assert (np.abs(g[k] - ref[k])[at] / floor[at]).max(initial=0.0) < TOL["f32"], k
            if k != "dV":
                assert not np.isfinite(g[k][~rows]).all(axis=-1).any(), k
        if which == "dO":
            assert not np.isfinite(g["dV"][i <= ROW if causal else i >= 0, COL]).any()
