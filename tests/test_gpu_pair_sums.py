"""GPU: the sums of the CUDA-core kernels are as good at every scale of their operands.

The statistics, normalisers and feature gradients are sums of cancelling terms, carried as pairs of floats and
rounded once.  How many bits such a sum keeps must depend on its own terms alone, not on what else its tile holds.
"""
import math

import numpy as np
import pytest

from cases import Case, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


def _case(n, d, dv, M, L, causal, seed):
    return Case(1, 2, n, d, M, L, "f32", causal, seed=seed, qkv_scale=1.0 / math.sqrt(d), dv=dv, with_grad=True)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("n,d,dv,M,L", [(150, 32, 32, 8, 8), (200, 64, 96, 8, 8), (70, 20, 33, 3, 5)])
def test_sums_do_not_depend_on_other_columns(n, d, dv, M, L, causal):
    """Columns of V scaled by 2^-18 and 2^-6 with the columns of dO scaled by the inverse: every product of a column
    of V and one of dO, and every power of two, stays exact, so dQ and dK keep their bits, and so do O and dV
    after their own scale."""
    case = _case(n, d, dv, M, L, causal, 211)
    lu = case.luna()
    O, g = case.run_fwd(lu), case.run_bwd(lu)
    plain = {"O": to_host(O), **{k: to_host(g[k]) for k in ("dQ", "dK", "dV")}}
    import torch
    scale = torch.tensor([2.0 ** (-18, 0, -6)[c % 3] for c in range(dv)], dtype=torch.float32, device="cuda")
    case.dev["V"] = case.dev["V"] * scale
    case.dev["dO"] = case.dev["dO"] / scale
    O, g = case.run_fwd(lu), case.run_bwd(lu)
    s = to_host(scale)
    got = {"O": to_host(O) / s, "dQ": to_host(g["dQ"]), "dK": to_host(g["dK"]), "dV": to_host(g["dV"]) * s}
    for k, v in plain.items():
        assert np.array_equal(got[k], v), (k, int((got[k] != v).sum()))


def test_streaming_outputs_are_no_further_off_than_fp64_sums():
    """fp32 outputs and dV of the streaming form.  Sums in fp64 over tiles of 16 rows, with fp32 scores, measured at
    this shape: O 6.2e-8 and dV 1.15e-7 of the tensor's rms away from the oracle (root mean square; 16 seeds, which
    differ by a few per cent).  The gates are these figures and a tenth."""
    err = {"O": [], "dV": []}
    for seed in range(4):
        case = _case(300, 64, 64, 8, 8, True, 223 + seed)
        lu = case.luna()
        got = {"O": to_host(case.run_fwd(lu)), "dV": to_host(case.run_bwd(lu)["dV"])}
        ref = {"O": case.oracle_fwd(), "dV": case.oracle_bwd()["dV"]}
        for k in err:
            err[k].append(math.sqrt(np.mean((got[k] - ref[k]) ** 2) / np.mean(ref[k] ** 2)))
    assert np.mean(err["O"]) < 6.8e-8 and np.mean(err["dV"]) < 1.27e-7, err


@pytest.mark.parametrize("causal", [False, True])
def test_projection_gradients_are_the_sums_of_their_rows(causal):
    """With W the identity, dX = dU W returns each row's dU, so dW = sum_rows dU x^T and db = sum_rows dU over Q and K
    can be formed on the host in 64 bits from the call's own dQ and dK.  Half an ulp for the result's rounding, and
    2^-42 of the terms' sizes for the pairs: their low parts are sums of at most 500 roundings of 2^-25, rounded at
    2^-25 in turn (sqrt(500) 2^-50 of the sizes if these are independent), and a margin of eight."""
    import synth
    d, n = 8, 500
    params = synth.phi_params(227, d, d, 8, 64)
    params["W"], params["b"] = np.eye(d, dtype=np.float32), np.zeros(d, np.float32)
    case = Case(2, 2, n, d, d, 8, "f32", causal, seed=227, params=params, with_grad=True)
    lu = case.luna()
    case.run_fwd(lu)
    g = {k: to_host(v) for k, v in case.run_bwd(lu).items()}
    x = {k: case.inp[k].value.reshape(-1, d) for k in ("Q", "K")}
    du = {k: g["d" + k].reshape(-1, d) for k in ("Q", "K")}
    for key, ref, size in (("dW", sum(du[k].T @ x[k] for k in x), sum(abs(du[k]).T @ abs(x[k]) for k in x)),
                           ("db", sum(du[k].sum(0) for k in x), sum(abs(du[k]).sum(0) for k in x))):
        half_ulp = np.spacing(abs(g[key]).astype(np.float32)).astype(np.float64) / 2
        assert (abs(g[key] - ref) <= half_ulp + 2.0 ** -42 * size).all(), key
