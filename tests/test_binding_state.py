"""The binding's place of the final state (no GPU): it follows the descriptors that the object holds now."""
import pytest


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")  # noqa: F841
    from paper_2512_08061_gb300 import build
    build.build()
    import paper_2512_08061_gb300.luna as L
    return L


def _decoded(L, lu, monkeypatch):
    """Arguments S, S_stride, z, z_stride of the decode call."""
    import torch
    got = []
    monkeypatch.setattr(L, "luna_attn_decode", lambda *a: got.append(a[7:11]))
    q = torch.zeros(lu.ad.B, lu.ad.H, lu.ad.d)
    lu.decode(q, q, torch.zeros(lu.ad.B, lu.ad.H, lu.ad.dv))
    return got[0]


def test_decode_follows_changed_descriptors(L, monkeypatch):
    """One object serves shorter sequences, fewer heads or another feature map by a new descriptor, or by a field of
    the one it has; the state it decodes from is where luna_state_final puts it for these."""
    import torch
    lu = L.Luna(2, 2, 3000, 16, 16, 4, 4, 8, True, 1e-6, torch.float32, device="cpu")
    check = lambda: _decoded(L, lu, monkeypatch) == L.luna_state_final(lu.ad, lu.pd, lu.state)  # noqa: E731
    assert check() and check()
    lu.ad.n = 200
    assert check()
    lu.ad = L.attn_desc(1, 2, 100, 16, 8, True, 0, 1e-6, 0)
    assert check()
    lu.pd = L.phi_desc(2, 4, 8)
    assert check()
    lu.state = torch.empty_like(lu.state)
    assert check()
    lu.ad.causal = 0
    with pytest.raises(L.LunaError) as e:
        check()
    assert e.value.status == 1


def test_first_decode_looks_nothing_up(L, monkeypatch):
    """The place of the state is found with the object, not by its first decode step."""
    lu = L.Luna(1, 2, 100, 16, 16, 4, 4, 8, True, 1e-6, device="cpu")
    monkeypatch.setattr(L, "luna_state_final", lambda *a: pytest.fail("looked up in the decode call"))
    _decoded(L, lu, monkeypatch)
