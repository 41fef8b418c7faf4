"""Embedding gradient from sorted token runs: run lengths on both sides of the block / warp split, several sort chunks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import Model  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,V,hot", [
    (1, 1, 64, 0),            # one position
    (1, 23, 64, 23), (1, 24, 64, 24), (1, 25, 64, 25),     # one run just below, at and above the split
    (3, 171, 512, 100),       # a long run among short ones, ragged sort size
    (5, 1639, 700, 3000),     # two sort chunks: tokens that occur in both are added to in chunk order
])
def test_embedding_gradient_sums_token_rows(B, T, V, hot):
    rng = np.random.default_rng(B * T)
    tok = rng.integers(0, V, size=(B, T)).astype(np.int32)
    flat = tok.reshape(-1)
    flat[rng.permutation(flat.size)[:hot]] = 7
    m = Model(1, 1, 128, 4, 256, V, 1, B, T, attn_bwd="two_kernels")
    for name in m.names:
        m.set_param(name, (rng.standard_normal(m.shapes[name]) * 0.05 + (1.0 if name.endswith(".g") else 0.0)).astype(np.float32))
    runs = []
    for _ in range(2):
        m.train_step(tok, rng.integers(0, V, size=(B, T)).astype(np.int32) if not runs else runs[0][2])
        m.sync()
        runs.append((m.get_grad("wte"), m.get_grad("wpe"), m._keep[1]))
    wte, wpe, _ = runs[0]
    assert np.array_equal(wte, runs[1][0]) and np.array_equal(wpe, runs[1][1])
    # the position gradient is the same rows summed over the batch, so the totals agree; rows no token selects are zero
    unused = np.setdiff1d(np.arange(V), flat)
    assert not wte[unused].any()
    # with one sequence every position's row is a row of the position gradient
    if B == 1:
        ref = np.zeros((V, 128))
        np.add.at(ref, flat, wpe[:T].astype(np.float64))
        # fp32 sums of at most 25 rows
        assert np.linalg.norm(wte - ref) <= 25 * 2.0 ** -24 * np.linalg.norm(np.abs(ref)) + 1e-12
    a, b = wte.astype(np.float64).sum(0), wpe.astype(np.float64).sum(0)
    scale = np.abs(wpe.astype(np.float64)).sum(0)
    assert np.all(np.abs(a - b) <= flat.size * 2.0 ** -24 * np.maximum(scale, np.abs(wte.astype(np.float64)).sum(0)) + 1e-12)
