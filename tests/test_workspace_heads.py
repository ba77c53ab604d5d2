"""The backward workspace of a problem with many heads holds what the kernels use."""
import pytest


@pytest.fixture(scope="module")
def L():
    from paper_2512_08061_gb300 import build
    build.build()
    import paper_2512_08061_gb300.luna as lib
    return lib


@pytest.mark.parametrize("n,d,dv,M,Lc", [(512, 64, 64, 8, 8), (33, 20, 96, 3, 5), (4096, 128, 128, 16, 8)])
def test_one_range_per_head_takes_one_partial(L, n, d, dv, M, Lc):
    """With a block or more per SM from the heads alone, every head is one range in each pass: its statistics and
    their gradients take one partial and one sum each, [D][dv] and [D] floats, beside two rows of fp64 parameter
    gradients, two counters and two words of the work split.  (Buffers start at multiples of 256 bytes.)"""
    pd, hid, heads = L.phi_desc(M, Lc, 64), 64, 1300
    size = [L.luna_workspace_size(L.attn_desc(1, h, n, d, dv, io=L.LUNA_F32), pd, True) for h in (heads, 2 * heads)]
    D = M * Lc
    grads = M * d + M + (Lc * hid + 1) * Lc * 2  # dW, db and the interval histogram of every channel
    per_head = 4 * 4 * (D * dv + D) + 2 * 8 * grads + 4 * 4
    assert abs(size[1] - size[0] - heads * per_head) <= 16 * 256
