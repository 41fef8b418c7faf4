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


def test_forward_beside_another_streams_traffic():
    """Many launches while another stream keeps the memory and the SMs busy: no warp may miss a barrier phase however late it
    comes to wait for it (a CTA whose wait runs out leaves its later items unwritten)."""
    B, T, H, dh = 5, 501, 16, 32                     # two items for some of the CTAs
    d = H * dh
    qkv = torch.randn(B * T, 3 * d, device=DEV).to(torch.bfloat16)
    big = torch.zeros(64 << 20, device=DEV)
    outs = [torch.zeros(B * T, d, device=DEV, dtype=torch.bfloat16) for _ in range(2)]
    lse = torch.zeros(B, H, T, device=DEV)
    il.op_attention_fwd(qkv, outs[0], lse, B, T, H, dh)
    torch.cuda.synchronize()
    ref = outs[0].clone()
    side = torch.cuda.Stream()
    for _ in range(40):
        with torch.cuda.stream(side):
            for _ in range(4):
                big.add_(1.0)
        for i in range(50):
            outs[1].fill_(7.0)
            il.op_attention_fwd(qkv, outs[1], lse, B, T, H, dh, stream=torch.cuda.current_stream().cuda_stream)
        assert torch.equal(outs[1], ref)
    torch.cuda.synchronize()
