"""GPU: the streaming form on tensor cores (bf16, d = dv = 128, M = 16): its workspace, and the paths that the
alignment of the caller's tensors and the number of heads select."""
import math

import pytest

from cases import TOL, Case, guarded_bytes, check_guards, relerr, relerr_rows, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_08061_gb300 import build
    build.build()


def _case(B, H, n, **kw):
    return Case(B, H, n, 128, 16, 8, "bf16", True, seed=251, qkv_scale=1.0 / math.sqrt(128), **kw)


def _shifted(t, elems):
    """A copy of t that starts `elems` elements after a 256-byte boundary."""
    import torch
    buf = torch.empty(t.numel() + 128, dtype=t.dtype, device=t.device)
    out = buf[elems:elems + t.numel()].view(t.shape)
    out.copy_(t)
    return out


def test_workspace_holds_what_the_kernels_use():
    """Per row of a backward pass: dphi (fp32) and phi(k), phi(q)/den (bf16 hi and lo) of 128 features, and two floats
    of row statistics.  The number of segments (64) is the same for both lengths."""
    import paper_2512_08061_gb300.luna as L
    pd = L.phi_desc(16, 8, 64)
    size = [L.luna_workspace_size(L.attn_desc(1, 2, n, 128, 128, causal=True), pd, True) for n in (8192, 16384)]
    assert size[1] - size[0] == 2 * 8192 * (128 * 4 + 2 * 2 * 128 * 2 + 2 * 4)


@pytest.mark.parametrize("per_head", [False, True])
def test_unaligned_inputs_take_the_generic_backward(per_head):
    """Inputs that start 8 bytes off a 16-byte boundary cannot be loaded by TMA; the generic kernels, whose row
    statistics are larger, run in the same workspace (between guard bands)."""
    case = _case(2, 2, 330, with_grad=True, lengths=[330, 101], per_head=per_head)
    lu = case.luna()
    for k in ("Q", "K", "V", "dO"):
        case.dev[k] = _shifted(case.dev[k], 4)
    assert relerr_rows(to_host(case.run_fwd(lu)), case.oracle_fwd()) < TOL["bf16"]
    ref = case.oracle_bwd()
    for use_state in (True, False):
        g = case.run_bwd(lu, use_state=use_state)
        for k in ("dV", "dW", "dw1", "db1", "dw2", "db2"):
            assert relerr(to_host(g[k]), ref[k]) < TOL["bf16"], k


def test_outputs_at_a_16_byte_boundary():
    """O may start at any 16-byte boundary; its 32-byte stores are used only where the rows allow them."""
    import torch
    case = _case(1, 2, 300)
    lu = case.luna()
    O = case.run_fwd(lu)
    band = []
    raw = guarded_bytes(O.numel() * 2 + 16, O.device, band)
    shifted = raw[16:].view(torch.bfloat16).view(O.shape)
    lu.forward(case.dev["Q"], case.dev["K"], case.dev["V"], None, O=shifted)
    check_guards(band)
    assert torch.equal(shifted, O)


def test_one_segment_per_head_with_more_heads_than_blocks():
    """Sequences of one state segment: the key pass writes each head's state itself, also when a block holds several
    heads.  The same heads in calls of four give the same bits."""
    import torch
    import paper_2512_08061_gb300.luna as L
    H, n = 400, 100
    case = _case(1, H, n)
    lu = case.luna()
    O = case.run_fwd(lu)

    def states(l, heads):
        S, Ss, z, zs = L.luna_state_final(l.ad, l.pd, l.state)
        flat = l.state.view(torch.float32)
        at = [flat.storage_offset() + (p - l.state.data_ptr()) // 4 for p in (S, z)]
        return flat.as_strided((heads, 128 * 128), (Ss, 1), at[0]), flat.as_strided((heads, 128), (zs, 1), at[1])

    S, z = states(lu, H)
    part = L.Luna(1, 4, n, 128, 128, 16, 8, 64, True, case.eps, torch.bfloat16)
    part.prepare({k: torch.from_numpy(v).cuda() for k, v in case.params.items()})
    for h in range(0, H, 4):
        x = [case.dev[k][:, h:h + 4].contiguous() for k in ("Q", "K", "V")]
        assert torch.equal(part.forward(*x), O[:, h:h + 4])
        Sp, zp = states(part, 4)
        assert torch.equal(Sp, S[h:h + 4]) and torch.equal(zp, z[h:h + 4])
