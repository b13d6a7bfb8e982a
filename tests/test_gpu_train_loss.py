"""The training loss is the mean of squares formed and added in FP64."""
import ctypes

import numpy as np
import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("hidden,layers,replaced", [(64, 2, 1), (32, 1, 1), (64, 2, 2), (32, 3, 1)])
@pytest.mark.parametrize("B,T", [(16, 1), (144, 3)])
@pytest.mark.parametrize("top,spread", [(1.0, 0), (4e19, 0), (1e-4, 30), (1e-12, 6), (1e-20, 0)])
def test_loss_of_a_network_that_predicts_zero(hidden, layers, replaced, B, T, top, spread):
    """With all weights zero the error is the target itself, so the loss must be the
    FP64 mean of the squares to one FP32 rounding (6e-8, or half the smallest
    subnormal; the FP64 sum of at most 21,600 squares is off by less than 1e-11): for
    targets of unit size, for some of 4e19, whose squares exceed FP32's range while
    their mean does not, over 30 orders of magnitude (down to subnormal ones), and
    where the squares are subnormal in FP32."""
    dn = lib()
    ctx = dn.Context(level_solve=2, train_batch=B, train_seq=T, hidden=hidden, gru_layers=layers,
                     replaced_levels=replaced)
    k = 2 ** replaced + 1
    c_in, c_out = 4 * k * k + 4, 2 * k * k
    ctx.set_weights(torch.zeros(ctx.num_params()))
    rng = np.random.default_rng(B + T + hidden)
    X = torch.from_numpy(rng.standard_normal((B, T, c_in))).to(torch.bfloat16).cuda()
    y = rng.standard_normal((B, T, c_out)).astype(np.float32)
    if top < 1:
        y = (top * y * 10.0 ** rng.uniform(-spread, 0, y.shape)).astype(np.float32)
    y[0, 0, 3], y[B - 1, T - 1, c_out - 1] = top, -top
    Y = torch.from_numpy(y).cuda()
    loss = ctypes.c_float()
    ctx._check(ctx.lib.dnnmg_train_grad(ctx.h, X.data_ptr(), Y.data_ptr(), B, T, None,
                                        ctypes.byref(loss)))
    ref = float((y.astype(np.float64) ** 2).mean())
    assert abs(loss.value - ref) <= max(6e-8 * ref, 0.7e-45), (loss.value, ref)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
def test_loss_of_targets_that_are_not_finite(bad):
    dn = lib()
    B, T = 32, 2
    ctx = dn.Context(level_solve=2, train_batch=B, train_seq=T)
    ctx.set_weights(torch.zeros(ctx.num_params()))
    X = torch.zeros(B, T, 40, dtype=torch.bfloat16, device="cuda")
    Y = torch.ones(B, T, 18, device="cuda")
    Y[B - 1, 1, 17] = bad
    loss = ctypes.c_float()
    ctx._check(ctx.lib.dnnmg_train_grad(ctx.h, X.data_ptr(), Y.data_ptr(), B, T, None,
                                        ctypes.byref(loss)))
    assert np.isnan(loss.value) if np.isnan(bad) else loss.value == float("inf")


@pytest.mark.parametrize("B,T", [(16, 1), (16, 4)])
def test_loss_is_that_of_the_call(B, T):
    """The host reads the loss of the call it waits for, in short calls whose
    targets change from one to the next (zero weights: the mean of their squares)."""
    dn = lib()
    for _ in range(20):  # first calls of new contexts too
        ctx = dn.Context(level_solve=2, train_batch=B, train_seq=T)
        ctx.set_weights(torch.zeros(ctx.num_params()))
        X = torch.zeros(B, T, 40, dtype=torch.bfloat16, device="cuda")
        Y = [torch.full((B, T, 18), float(k), device="cuda") for k in range(1, 6)]
        torch.cuda.synchronize()
        loss = ctypes.c_float()
        for k in range(200):
            ctx._check(ctx.lib.dnnmg_train_grad(ctx.h, X.data_ptr(), Y[k % 5].data_ptr(), B, T, None,
                                                ctypes.byref(loss)))
            assert loss.value == (k % 5 + 1) ** 2, (k, loss.value)
