"""The model's passes on as many samples as their 32-bit count names: a block's
step past the last sample must end its loop, not start over at sample 0.  (The
samples take 120 GB; nearly all are zero, and equal samples have equal outputs.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
M = (1 << 32) - 1


def test_last_sample_ends_the_loop(gpu_lib):
    import torch

    t = gpu_lib
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 140e9:
        pytest.skip("needs 120 GB of free device memory")
    ctx = t.tkc_create()
    try:
        t.tkc_mlp_init(ctx, 5)
        w = t.tkc_get_source_model(ctx).copy()
        w[320:384] = np.linspace(-1, 1, 64)  # biases, so that a zero sample has an output
        w[4608] = 0.25
        t.tkc_set_source_model(ctx, w)
        ends = torch.randn(200, t.TKC_MLP_FEATURES, device="cuda")
        few = torch.cat([ends, torch.zeros(1, t.TKC_MLP_FEATURES, device="cuda")])
        want = torch.empty(201, device="cuda")
        t.tkc_mlp_forward(ctx, few, want)
        x = torch.zeros(M, t.TKC_MLP_FEATURES, device="cuda")
        x[:100], x[-100:] = ends[:100], ends[100:]
        y = torch.full((M,), float("nan"), device="cuda")
        t.tkc_mlp_forward(ctx, x, y)
        assert torch.equal(y[:100], want[:100]) and torch.equal(y[-100:], want[100:200])
        for a in range(100, M - 100, 1 << 30):
            part = y[a:min(a + (1 << 30), M - 100)]
            assert bool((part == want[200]).all())
        y.zero_()  # the targets
        grad = torch.full((t.TKC_MLP_PARAMS,), float("nan"), device="cuda")
        loss = t.tkc_mlp_gradient(ctx, x, y, grad)
        sq = want.double() ** 2
        mean = float((sq[:200].sum() + sq[200] * (M - 200)) / M)
        assert abs(loss - mean) <= 1e-6 * mean  # terms and sums in 64 bits, the result rounded to 32
        assert bool(torch.isfinite(grad).all()) and float(grad.abs().max()) > 0
    finally:
        x = y = None
        torch.cuda.empty_cache()
        t.tkc_destroy(ctx)
