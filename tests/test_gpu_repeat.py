"""GPU: what the CUDA-core kernels repeat bit for bit.

O, dQ, dK, dV, dW and db are sums in a fixed order.  (The channel MLPs' gradients come from histograms filled by
reductions whose order varies in the last bits of their fp64 sums.)
"""
import math

import pytest

from cases import Case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("d,M,L,per_head", [(64, 8, 8, False), (20, 3, 5, False), (32, 8, 8, True)])
def test_repeated_backward_keeps_its_bits(d, M, L, per_head, causal):
    """The second sequence is the first with dO negated, so that its rows of dU are the first's negated but for
    roundings: dW and db cancel to a few last bits, and any other order of their sums shows."""
    import torch
    case = Case(2, 4, 1000, d, M, L, "f32", causal, seed=241, qkv_scale=1.0 / math.sqrt(d), with_grad=True,
                per_head=per_head)
    lu = case.luna()
    for k, sign in (("Q", 1), ("K", 1), ("V", 1), ("dO", -1)):
        case.dev[k][1] = sign * case.dev[k][0]
    first = None
    for _ in range(20):
        O, g = case.run_fwd(lu), case.run_bwd(lu)
        got = {"O": O, **{k: g[k] for k in ("dQ", "dK", "dV", "dW", "db")}}
        if first is None:
            first = got
        for k, v in got.items():
            assert torch.equal(v, first[k]), (k, int((v != first[k]).sum()))
