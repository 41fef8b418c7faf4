"""Attention backward with sums of fixed order, every head dimension: short sequences (one 128 x 128 tile) at the edges of the
16-wide contraction steps and of the two 64-key halves, longer ones at the edges of the 128-row tiles and 64-wide sweep steps, more
items than resident CTAs."""
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import binding as il  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dh", [32, 64, 80, 128, 256])
@pytest.mark.parametrize("NB,B,T,H", [(1, 1, 2, 1), (2, 1, 15, 3), (2, 2, 16, 2), (4, 2, 17, 2), (3, 3, 63, 4), (2, 1, 64, 2), (2, 2, 65, 3),
                                      (1, 1, 113, 2), (2, 1, 127, 2), (160, 80, 128, 4), (301, 301, 40, 1),
                                      (2, 1, 129, 2), (2, 2, 192, 1), (1, 1, 193, 3), (1, 1, 256, 2), (3, 1, 257, 2), (40, 20, 320, 4),
                                      (2, 1, 1100, 3)])
def test_backward_matches_fp64(NB, B, T, H, dh):
    g = torch.Generator(device=DEV)
    g.manual_seed(NB * T + dh)
    d = H * dh
    qkv = torch.randn(B * T, 3 * d, device=DEV, generator=g).to(torch.bfloat16)
    dout = torch.randn(NB * T, d, device=DEV, generator=g).to(torch.bfloat16)
    q, k, v = (x.permute(0, 2, 1, 3).double() for x in qkv.view(B, T, 3, H, dh).unbind(2))
    s = (q @ k.transpose(-1, -2)) / dh ** 0.5
    s = s.masked_fill(torch.ones(T, T, device=DEV, dtype=torch.bool).triu(1), float("-inf"))
    lse = torch.logsumexp(s, -1)
    idx = torch.arange(NB, device=DEV) % B
    p = torch.softmax(s, -1)[idx]
    do = dout.view(NB, T, H, dh).permute(0, 2, 1, 3).double()
    dp = do @ v[idx].transpose(-1, -2)
    ds = p * (dp - (p * dp).sum(-1, keepdim=True)) / dh ** 0.5
    ref = torch.stack([ds @ k[idx], ds.transpose(-1, -2) @ q[idx], p.transpose(-1, -2) @ do])        # [3, NB, H, T, dh]
    ref = ref.permute(1, 3, 0, 2, 4).reshape(NB * T, 3 * d)
    got = torch.full((NB * T, 3 * d), 7.0, device=DEV, dtype=torch.bfloat16)
    o = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3).reshape(B * T, d).to(torch.bfloat16)
    delta = torch.zeros(NB * H * T, device=DEV)
    il.op_attention_bwd(qkv, o, lse.float(), dout, got, delta, NB, B, T, H, dh)
    torch.cuda.synchronize()
    for i in range(3):
        a, b = got[:, i * d:(i + 1) * d].double(), ref[:, i * d:(i + 1) * d]
        # P or dS, the result and (in the row sums of longer sequences) O are rounded to bf16, 2^-9 / sqrt(3) each in the
        # mean: together 2^-9
        assert float((a - b).norm() / b.norm()) < 2.0 ** -8, "qkv"[i]
    again = torch.full((NB * T, 3 * d), -3.0, device=DEV, dtype=torch.bfloat16)
    il.op_attention_bwd(qkv, o, lse.float(), dout, again, delta, NB, B, T, H, dh)
    torch.cuda.synchronize()
    assert torch.equal(got, again)                # every sum has a fixed order


@pytest.mark.parametrize("dh", [32, 64])
@pytest.mark.parametrize("NB,B,T,H", [(40, 20, 320, 4), (3, 3, 257, 60), (16, 8, 501, 16), (151, 151, 129, 1), (2, 1, 2049, 12)])
def test_one_sweep_with_several_items_per_cta(NB, B, T, H, dh):
    """More (key tile, sequence, head) items than SMs, of several lengths: K / V, accumulators, rings and step counters go from
    item to item.  Against the fixed-order form (above against fp64): dK and dV bit for bit, dQ, whose share of every key tile
    has the same bits there and here, up to the order of their fp32 sum and one rounding to bf16."""
    g = torch.Generator(device=DEV)
    g.manual_seed(NB + T + dh)
    d = H * dh
    qkv = torch.randn(B * T, 3 * d, device=DEV, generator=g).to(torch.bfloat16)
    dout = torch.randn(NB * T, d, device=DEV, generator=g).to(torch.bfloat16)
    o, lse = torch.empty(B * T, d, device=DEV, dtype=torch.bfloat16), torch.empty(B, H, T, device=DEV)
    il.op_attention_fwd(qkv, o, lse, B, T, H, dh)
    delta, acc = torch.empty(NB * H * T, device=DEV), torch.full((NB * T, d), 9.0, device=DEV)
    two = torch.empty(NB * T, 3 * d, device=DEV, dtype=torch.bfloat16)
    il.op_attention_bwd(qkv, o, lse, dout, two, delta, NB, B, T, H, dh)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    one = torch.empty_like(two)
    a = torch.randn(1024, 1024, device=DEV, dtype=torch.bfloat16)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for attempt in range(6):
        one.fill_(5.0)
        if attempt % 2:                           # beside kernels of another stream
            with torch.cuda.stream(side):
                for _ in range(20):
                    a @ a
        il.op_attention_bwd_one_sweep(qkv, o, lse, dout, one, delta, acc, NB, B, T, H, dh, err_word=err)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        assert torch.equal(one[:, d:], two[:, d:])
        x, y = (t[:, :d].float().view(NB, T, H, dh).permute(0, 2, 1, 3) for t in (one, two))
        for t0 in range(0, T, 128):               # tile by tile: one that missed a share is not lost among the others
            num, den = ((x - y)[:, :, t0:t0 + 128].norm(dim=(-1, -2)), y[:, :, t0:t0 + 128].norm(dim=(-1, -2)))
            assert bool((num <= 2.0 ** -8 * den).all()), (attempt, t0)
