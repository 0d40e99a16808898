"""The tcgen05 convolutions, input gradients and weight gradients at the edges
of their strips: both poles in one strip, a last strip of one, two or four
rows, levels that the kernel takes and levels that it does not, and more strips
than a block's first one.  Same bars as test_gpu_cnn.py."""
import numpy as np
import pytest

from oracle import cnn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402
from test_gpu_cnn import dev, inputs, model_with, params, rel  # noqa: E402


@pytest.mark.parametrize("B,H,W", [(1, 8, 512), (1, 20, 512), (2, 12, 256), (1, 36, 128), (12, 64, 256), (4, 24, 64),
                                   (1, 12, 768)])
def test_forward_and_gradients(B, H, W):
    P = params(70 + H)
    m = model_with(P)
    x0 = cnn.round_bf16(inputs(80 + H, B, H, W))
    if B > 2:                        # (even) samples alternate, so that the oracle runs two
        x0 = np.ascontiguousarray(x0[np.arange(B) % 2])
    target = np.random.default_rng(90 + H).standard_normal((B, H, W))[np.arange(B) % 2 if B > 2 else slice(None)]
    y = torch.empty((B, H, W), dtype=torch.float32, device="cuda")
    sw.sw_model_forward(m, dev(x0), y)
    _, g = sw.sw_model_loss_grad(m, dev(x0), dev(target))
    yg = y.cpu().numpy()
    Pr = {k: (cnn.round_bf16(v) if k.endswith(".w") else v) for k, v in P.items()}
    Gr, n = None, min(B, 2)
    for b in range(n):
        yo, cache = cnn.forward(P, x0[b], bf16=True)
        for q in range(b, B, n):
            assert rel(yg[q], yo) <= 1e-2
        gb = cnn.backward(Pr, cache, 2.0 * (yo - target[b]))
        Gr = gb if Gr is None else {k: Gr[k] + gb[k] for k in Gr}
    Gg = cnn.unflatten_params(g.astype(np.float64))
    for name, _, _, _ in cnn.LAYERS:
        for part in (".w", ".b"):
            assert rel(Gg[name + part], Gr[name + part] / (n * H * W)) <= 2.5e-2, name + part
