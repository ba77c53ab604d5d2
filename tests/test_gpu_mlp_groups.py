"""GPU: parameter gradients of non-ReLU channel MLPs, whose hidden units are spread over a block's threads in groups:
unit counts that leave a remainder of the block, one group, and fewer samples than groups.  Tolerance: the fp32 parity
gate of the other GPU tests (1e-4 of the oracle, floored at the tensor's rms)."""
import math

import pytest

from cases import TOL, Case, relerr, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("M,L,hidden,shared,n", [(8, 8, 64, True, 150), (3, 5, 100, True, 77), (8, 16, 5, True, 64),
                                                 (2, 3, 7, False, 33), (8, 16, 32, False, 65), (4, 4, 128, True, 3)])
def test_unit_groups(M, L, hidden, shared, n, causal):
    case = Case(1, 2, n, 32, M, L, "f32", causal, seed=251, qkv_scale=1.0 / math.sqrt(32), hidden=hidden,
                with_grad=True, shared=shared, act="tanh")
    lu = case.luna()
    case.run_fwd(lu)
    g, ref = case.run_bwd(lu), case.oracle_bwd()
    for k in ("dw1", "db1", "dw2", "db2"):
        assert relerr(to_host(g[k]), ref[k]) < TOL["f32"], k

