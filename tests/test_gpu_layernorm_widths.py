"""LayerNorm backward inside the blocks at widths on both sides of its layouts: a ragged last 128 columns, one, two and four warps
per row, more rows than the grid holds at once, stacked gradient streams.  Checked through the step against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import il_oracle as orc  # noqa: E402
from paper_2010_04116_b200 import Model  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,dh,B,T", [(1, 32, 2, 9), (5, 32, 1, 200), (13, 80, 1, 40), (31, 32, 3, 11), (1, 128, 1, 1300), (16, 80, 2, 17),
                                      (33, 32, 1, 700), (64, 32, 1, 5), (65, 32, 2, 10), (24, 128, 1, 6)])
def test_parameter_and_bias_gradients(H, dh, B, T):
    d, F, V, K, Lc, n = H * dh, 64, 96, 3, 2, 2
    rng = np.random.default_rng(d + T)
    m = Model(K, Lc, d, H, F, V, n, B, T, attn_bwd="two_kernels")
    P = {name: rng.standard_normal(m.shapes[name]) * 0.02 + (1.0 if name.endswith(".g") else 0.0) for name in m.names}
    P = {name: p.astype(np.float32) for name, p in P.items()}
    for name in m.names:
        m.set_param(name, P[name])
    tok, tgt = (rng.integers(0, V, size=(B, T)).astype(np.int32) for _ in range(2))
    m.train_step(tok, tgt)
    m.sync()
    _, G = orc.nwise_gradients(P, tok, tgt, K, Lc, H, n)
    for name in m.names:
        if name.startswith("c") and (name.endswith((".g", ".b", ".bo", ".b2", "wqkv")) or name.endswith("b1")) or name in ("wte", "wpe"):
            ref = G[name]
            assert np.linalg.norm(m.get_grad(name) - ref) < 2e-2 * np.linalg.norm(ref), name       # bf16 operands, as for the whole step
