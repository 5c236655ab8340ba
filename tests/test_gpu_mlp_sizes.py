"""Batch forward and gradient of the predictor at the edges of its tiling.

A tile holds at most 64 samples in rows of four, the launch takes tiles of
equal size over 152 SMs, and a CTA adds up sums of 32 samples; so: one sample,
both sides of four, of 32 and of 64, of one tile of four per SM, of one full
tile per SM, and a size that leaves a last round nearly empty.

Tolerances against FP64 with the same BF16-rounded weights.  A hidden unit
is a sum of at most 64 products: its error is about sqrt(64) roundings of
2^-24 of terms that are O(1) against the largest, 5e-7 a layer and 2e-6 through
four layers, forward; backward the same again, with the samples' sum.  Ten
times that: 2e-5 forward and 4e-5 for a gradient, of the largest entry.
"""
import numpy as np
import pytest

import predictor_nets as PN
from test_gpu_predictor import dev, random_params

pytestmark = pytest.mark.gpu

SIZES = [1, 3, 4, 5, 31, 33, 63, 64, 65, 152 * 4 - 1, 152 * 4 + 1, 152 * 64 - 3, 152 * 64 + 1, 30000]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return torch, native


@pytest.mark.parametrize("n", SIZES)
def test_forward_and_gradient(env, orc, n):
    torch, native = env
    p = random_params(n)
    rng = np.random.default_rng(1000 + n)
    X = rng.normal(0, 1, (n, 40)).astype(np.float32)
    Y = rng.normal(0, 1, (n, 2)).astype(np.float32)
    pd, Xd, Yd = dev(torch, p), dev(torch, X), dev(torch, Y)
    out = torch.full((n + 1, 2), 7.0, dtype=torch.float32, device="cuda")  # the last row is not written
    assert native.cp_mlp_forward(pd.data_ptr(), Xd.data_ptr(), n, out.data_ptr()) == native.OK
    got = out.cpu().numpy().astype(np.float64)
    assert (got[n] == 7.0).all()
    want = orc.mlp_forward(p, X.astype(np.float64))
    np.testing.assert_allclose(got[:n], want, rtol=0, atol=2e-5 * np.abs(want).max())
    g = torch.empty(PN.NP, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    work = torch.full((native.cp_mlp_work_floats(),), float("nan"), dtype=torch.float32, device="cuda")
    assert native.cp_mlp_loss_grad(pd.data_ptr(), Xd.data_ptr(), Yd.data_ptr(), n, g.data_ptr(),
                                   loss.data_ptr(), work.data_ptr()) == native.OK
    want_loss, want_g = orc.mlp_loss_grad(p, X.astype(np.float64), Y.astype(np.float64))
    assert loss.item() == pytest.approx(want_loss, rel=4e-5)
    got_g = g.cpu().numpy().astype(np.float64)
    for name, size in (("W1", 2560), ("b1", 64), ("W2", 4096), ("b2", 64), ("W3", 4096), ("b3", 64),
                       ("W4", 128), ("b4", 2)):
        sl = slice(PN.OFF[name], PN.OFF[name] + size)
        np.testing.assert_allclose(got_g[sl], want_g[sl], rtol=0, atol=4e-5 * np.abs(want_g[sl]).max(),
                                   err_msg=name)
