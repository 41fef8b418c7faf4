"""Attention forward at the edges of its tiles (128-row tiles in pairs, 64-key halves) and of its dispatch (160 positions)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import binding as il  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dh", [32, 64, 80, 128])
@pytest.mark.parametrize("B,T,H", [(1, 160, 2), (2, 161, 1), (1, 191, 3), (1, 255, 2), (2, 256, 2), (1, 257, 2), (3, 384, 5), (1, 385, 2),
                                   (1, 1100, 3), (40, 300, 4)])
def test_forward_matches_fp64(B, T, H, dh):
    g = torch.Generator(device=DEV)
    g.manual_seed(B * T + dh)
    d = H * dh
    # one row's scores grow along the keys, so that the reference maximum has to be raised in mid-sweep
    qkv = (torch.randn(B * T, 3 * d, device=DEV, generator=g) * 1.5)
    qkv[:, d:2 * d] *= torch.linspace(0.2, 6.0, T, device=DEV).repeat(B)[:, None]
    qkv = qkv.to(torch.bfloat16)
    o = torch.full((B * T, d), 7.0, device=DEV, dtype=torch.bfloat16)
    lse = torch.full((B, H, T), 7.0, device=DEV)
    il.op_attention_fwd(qkv, o, lse, B, T, H, dh)
    torch.cuda.synchronize()
    q, k, v = (x.permute(0, 2, 1, 3).double() for x in qkv.view(B, T, 3, H, dh).unbind(2))
    s = (q @ k.transpose(-1, -2)) / dh ** 0.5
    s = s.masked_fill(torch.ones(T, T, device=DEV, dtype=torch.bool).triu(1), float("-inf"))
    ref = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3).reshape(B * T, d)
    # P and O are rounded to bf16: relative error 2^-9 / sqrt(3) each, and P's does not average out where one key dominates
    assert float((o.double() - ref).norm() / ref.norm()) < 2.0 ** -8
    rows = (o.double() - ref).norm(dim=1) / ref.norm(dim=1)
    assert float(rows.max()) < 2.0 ** -6                      # no single row is off by more than a few roundings
    assert float((lse.double() - torch.logsumexp(s, -1)).abs().max()) < 2e-4      # ex2.approx and fp32 sums at |lse| up to ~100
