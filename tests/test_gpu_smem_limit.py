"""GPU: shapes whose row tiles come out within the kernels' own static shared memory of the 227 KB limit.

The tile rule counts the arrays of a tile; a launch is refused when these and the static part together exceed the
limit, so a tile that fits by itself must still leave room.
"""
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


@pytest.mark.parametrize("M,L,hidden,d,dv,causal", [
    (3, 16, 8, 128, 128, True), (7, 8, 64, 40, 120, True), (12, 10, 48, 80, 112, False), (28, 2, 8, 64, 128, True),
    (29, 1, 32, 128, 128, True), (21, 2, 8, 128, 128, True), (32, 2, 16, 32, 128, True)])
def test_tiles_at_the_limit(M, L, hidden, d, dv, causal):
    case = Case(1, 1, 70, d, M, L, "f32", causal, seed=239, qkv_scale=1.0 / math.sqrt(d), hidden=hidden, dv=dv,
                with_grad=True)
    lu = case.luna()
    O = to_host(case.run_fwd(lu))
    g = case.run_bwd(lu)
    assert relerr(O, case.oracle_fwd()) < TOL["f32"]
    assert relerr(to_host(g["dV"]), case.oracle_bwd()["dV"]) < TOL["f32"]
