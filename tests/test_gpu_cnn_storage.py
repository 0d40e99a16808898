"""The network's buffers: what a batch needs and no more, and batches of other
sizes on one model."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402
from test_gpu_cnn import dev, inputs, model_with, params  # noqa: E402


def batch(B, H, W):
    return dev(inputs(90 + W, B, H, W)), dev(np.random.default_rng(91 + W).standard_normal((B, H, W)))


def test_no_storage_for_concatenations_that_are_not_stored():
    B, H, W = 32, 128, 256
    x0, t = batch(B, H, W)
    sw.sw_model_train_step(model_with(params(92)), x0[:1, :, :, :].contiguous(), t[:1].contiguous(), lr=1e-3)
    m = model_with(params(92))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sw.sw_model_train_step(m, x0, t, lr=1e-3)
    used = free - torch.cuda.mem_get_info()[0]
    # per point of the batch: 244 BF16 and 61 FP32 values, counted over the levels;
    # one sample's inputs and output in FP32
    need = B * H * W * (244 * 2 + 61 * 4) + 5 * H * W * 4
    assert need <= used <= need + (8 << 20)


def test_one_model_on_batches_of_other_sizes():
    """nx = 64 stores the middle level's concatenation, the others do not: each
    gives on a model that has run the others what it gives on a new one."""
    p = params(93)
    sizes = [(2, 16, 256), (3, 24, 64), (1, 8, 128), (9, 32, 64), (2, 16, 256), (3, 24, 64)]
    m = model_with(p)
    for B, H, W in sizes:
        x0, t = batch(B, H, W)
        got, want = (torch.empty((B, H, W), device="cuda") for _ in range(2))
        sw.sw_model_forward(m, x0, got)
        sw.sw_model_forward(model_with(p), x0, want)
        assert torch.equal(got, want)
        (la, ga), (lb, gb) = (sw.sw_model_loss_grad(q, x0, t) for q in (m, model_with(p)))
        # sums of the blocks' parts by FP32 atomics, in any order
        assert abs(la - lb) <= 1e-12 * lb
        assert np.linalg.norm(ga - gb) <= 1e-5 * np.linalg.norm(gb)
