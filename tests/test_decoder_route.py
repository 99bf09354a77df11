"""Which calls GqlaDecoder.absorb_step chains, by shape and slot count (no GPU: the library's calls are replaced by a recorder)."""
import pytest
import torch

from paper_2605_15250_b200 import binding as B
from paper_2605_15250_b200 import build as gbuild
from paper_2605_15250_b200 import decoder


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


def _tail(monkeypatch, slots, dtype=torch.bfloat16, fused_tail=True, **dims):
    calls = []
    for name in ("gqla_absorb_q", "gqla_decode_absorb", "gqla_combine_up_proj", "gqla_combine_splits", "gqla_up_proj"):
        monkeypatch.setattr(B, name, lambda *a, name=name: calls.append(name))
    d = dict(dict(h_q=128, g=8, d_h=128, r_kv=512, d_r=64), **dims)
    dec = object.__new__(decoder.GqlaDecoder)  # __init__ asks for CUDA tensors
    dec.dims = B.make_dims(**d)
    dec.__dict__.update(d, dtype=dtype, device="cpu", _buf={}, block_table=None, w_uk=None, w_uv=None, cache=None, seq_start=None,
                        seqlens=None, scale=1.0, status=None)
    q = [torch.zeros((2, 1, d["h_q"], n), dtype=dtype) for n in (d["d_h"], d["d_r"])]
    dec.absorb_step(*q, -slots, fused_tail=fused_tail)
    return calls[2:]


FUSED, SEPARATE = ["gqla_combine_up_proj"], ["gqla_combine_splits", "gqla_up_proj"]


@pytest.mark.parametrize("slots", [2, 4, 5, 12, 13])
def test_tail_of_the_absorb_step(monkeypatch, slots):
    """Five to twelve slots take the fused merge + up-projection where its tensor-core kernel covers the shape, and in fp32."""
    few, some = slots <= 4, slots <= 12
    for dims in (dict(), dict(h_q=28, g=4), dict(h_q=64, g=1), dict(r_kv=256), dict(dtype=torch.float32)):
        assert _tail(monkeypatch, slots, **dims) == (FUSED if some else SEPARATE), dims
    # 128 heads in one group, a wide latent row, dims of no tensor-core kernel
    for dims in (dict(g=1), dict(r_kv=1024), dict(r_kv=384)):
        assert _tail(monkeypatch, slots, **dims) == (FUSED if few else SEPARATE), dims
    assert _tail(monkeypatch, slots, fused_tail=False) == SEPARATE
