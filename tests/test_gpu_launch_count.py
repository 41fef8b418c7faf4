"""The number of kernels a model says it has launched, against a profiler's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import Model  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,d,H,V,B,T,attn_bwd", [
    (2, 256, 1, 9000, 2, 200, "two_kernels"),       # optimiser updates in parts, attention backward of head dimension 256
    (1, 128, 4, 512, 33, 256, "one_sweep"),         # embedding gradient of more positions than one sort holds
    (2, 128, 2, 300, 2, 40, "one_sweep"),           # short sequences
])
def test_launch_count(K, d, H, V, B, T, attn_bwd):
    rng = np.random.default_rng(1)
    m = Model(K, 1, d, H, 2 * d, V, K, B, T, attn_bwd=attn_bwd)
    for nm in m.names:
        m.set_param(nm, (rng.standard_normal(m.shapes[nm]) * 0.05 + nm.endswith(".g")).astype(np.float32))
    batch = [rng.integers(0, V, size=(B, T)).astype(np.int32) for _ in range(2)]
    for _ in range(3):                              # enqueued, recorded, replayed
        torch.cuda.synchronize()
        before = m.stats()[1]
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            m.train_step(*batch, adamw={"lr": 1e-3})
            torch.cuda.synchronize()
        kernels = [e for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA and not e.name.startswith("Mem")]
        assert m.stats()[1] - before == len(kernels)
    m.close()
