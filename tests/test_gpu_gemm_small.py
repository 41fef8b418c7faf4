"""Single-CTA GEMM tiles with the contraction split inside a cluster, against an fp64 product of the same bf16 operands."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import binding as il  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _case(M, N, K, layout, epi, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    a_mn, b_mn = layout

    def operand(rows, mn):
        t = torch.randn(rows, K, device=DEV, generator=g)
        m = t.t() if mn else t
        buf = torch.full((m.shape[0], (m.shape[1] + 7) // 8 * 8), 3.0, device=DEV, dtype=torch.bfloat16)
        buf[:, :m.shape[1]] = m
        e = buf[:, :m.shape[1]].double()
        return buf, (e.t() if mn else e)
    A, Ae = operand(M, a_mn)
    B, Be = operand(N, b_mn)
    return A, B, Ae @ Be.t(), g


@pytest.mark.parametrize("tile", [0, -1, -2, -4, -8, -65, -66, -68, -72])
@pytest.mark.parametrize("M,N,K,layout,epi", [
    (1, 8, 8, (0, 0), 0),              # one row, one slab: most of a cluster's k-ranges are empty
    (129, 130, 72, (0, 0), 1),         # one past a tile both ways, ragged last columns
    (128, 128, 1024, (0, 0), 2),       # exactly one tile
    (200, 196, 1003, (0, 1), 0),       # slabs not divisible by the split
    (300, 264, 520, (0, 1), 3),        # saved rows shared by stacked streams, column sums over the first stream
    (257, 72, 4104, (0, 1), 4),        # row factor
    (131, 260, 2505, (1, 1), 4),       # both operands MN-major, accumulating
])
def test_cluster_split_gemm(M, N, K, layout, epi, tile):
    A, B, ref, g = _case(M, N, K, layout, epi, M + N + K)
    ldc = (N + 7) // 8 * 8
    f32 = epi in (2, 4)
    out = torch.full((M, ldc), 2.0, device=DEV, dtype=torch.float32 if f32 else torch.bfloat16)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    kw, cs, act = {}, None, None
    if epi in (0, 1, 2):
        kw["bias"] = torch.randn(ldc, device=DEV, generator=g)
        ref = ref + kw["bias"][:N].double()
    if epi == 1:
        act = torch.zeros_like(out)
        kw["C2"] = act
        x = ref.requires_grad_()
        y = torch.nn.functional.gelu(x, approximate="tanh")
        ref, act_ref = torch.autograd.grad(y.sum(), x)[0], y.detach()
    elif epi == 2:
        kw["resid"] = torch.randn(M, ldc, device=DEV, generator=g)
        ref = ref + kw["resid"][:, :N].double()
    elif epi == 3:
        rows = (M + 1) // 2
        aux = torch.randn(rows, ldc, device=DEV, generator=g).to(torch.bfloat16)
        cs = torch.zeros(ldc, device=DEV)
        kw.update(aux=aux, ld_aux=ldc, aux_rows=rows, colsum=cs)
        ref = ref * aux.double()[torch.arange(M, device=DEV) % rows][:, :N]
    elif epi == 4 and layout == (0, 1):
        kw["rowscale"] = torch.rand(M, device=DEV, generator=g)
        ref = ref * kw["rowscale"].double()[:, None]
    elif epi == 4:
        kw["accumulate"] = 1
        ref = ref + 2.0
    il.op_gemm(M, N, K, A, A.shape[1], layout[0], B, B.shape[1], layout[1], epi, err, C_=out, ldc=ldc, tile_blocks=tile, **kw)
    torch.cuda.synchronize()
    assert int(err.item()) == 0

    def rel(a, b):
        return float((a.double() - b).norm() / b.norm())
    # fp32 sums: the tensor core truncates the running sum after every 16 products, on average by a quarter of 2^-23 of
    # its final magnitude and always towards zero, so K / 16 steps lose up to K / 16 * 2^-25, plus a few ulps for the
    # epilogue; bf16 results: half an ulp is 2^-9, and gelu' takes tanh.approx (absolute error 5e-4) on values of order one
    tol32 = K / 16 * 2.0 ** -25 + 2.0 ** -22
    tol = tol32 if f32 else (2.0 ** -9 if epi != 1 else 3e-3)
    assert rel(out[:, :N], ref) < tol
    if ldc > N:
        assert bool((out[:, N:] == 2.0).all())
    if act is not None:
        assert rel(act[:, :N], act_ref) < 3e-3
    if cs is not None:
        assert rel(cs[:N], ref[:(M + 1) // 2].sum(0)) < 4 * tol32


@pytest.mark.parametrize("tile", [-1, -8, -66, -3, -200, 7])
def test_tile_the_epilogue_does_not_have_is_chosen_from_the_shape(tile):
    """A tile_blocks that names no form of the product's epilogue and layout leaves the choice to the shape."""
    M, N, K = 130, 300, 72
    A, B, ref, g = _case(M, N, K, (0, 0), 5, 9)
    targets = torch.randint(0, N, (M,), device=DEV, generator=g).to(torch.int32)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    res = []
    for t in (0, tile):
        part = [torch.zeros(M, 3, device=DEV) for _ in range(2)]
        tgt = torch.zeros(M, device=DEV)
        il.op_gemm(M, N, K, A, A.shape[1], 0, B, B.shape[1], 0, 5, err, targets=targets, part_max=part[0], part_sum=part[1], part_ld=3,
                   tgt_logit=tgt, tile_blocks=t)
        torch.cuda.synchronize()
        res.append((*part, tgt))
    assert int(err.item()) == 0
    for x, y in zip(*res):
        assert torch.equal(x, y)
    # fp32 sums of 72 products, ex2.approx and the fp32 logarithm of sums near 300: a few ulps of values near ten each
    lse = (res[1][0].double() + res[1][1].double().log()).logsumexp(1)
    assert float((lse - ref.logsumexp(1)).abs().max()) < 1e-4
