"""The surrogate network's grouped products at the edges of their tiles: widths and batches
around the 32 x 32 (FP32) and 128 x 16 (BF16) tiles and the 64 / 128-deep slabs, widths that
forbid 16-byte loads, weight gradients summed in several parts of the batch, gathered rows;
forward, loss and every gradient against the FP64 oracle MLP."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu

# the network tests' tolerances: FP32 sums of at most ~1000 terms, 2^-24 each, well inside
# 2e-5 (outputs) and 1e-4 (gradients) of the scale; BF16 operands carry 2^-9 each
TOL = {"fp32": (2e-5, 1e-4), "bf16": (2e-2, 2e-2)}


@pytest.fixture(scope="module")
def kd():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2307_01571_gb300 import _build
    _build.build()
    from paper_2307_01571_gb300 import kd as mod
    return mod


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("widths,batch", [
    ([1, 1], 1), ([3, 33, 65, 2], 31), ([8, 32, 16, 4], 32), ([7, 129, 17, 5], 129),
    ([5, 64, 128, 4], 257), ([5, 256, 256, 256, 4], 1024), ([66, 130, 3], 515), ([4, 128, 20], 128)])
def test_products_at_tile_edges(kd, prec, widths, batch):
    rng = np.random.default_rng(len(widths) * 1000 + batch)
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.standard_normal((batch, widths[-1])).astype(np.float32)
    p = mlp.init_params(widths, 5)
    p = (p + 0.01 * rng.standard_normal(p.size)).astype(np.float32)     # biases too
    net = kd.MLP(widths)
    net.set_precision(kd.KD_MLP_BF16 if prec == "bf16" else kd.KD_MLP_FP32)
    net.set_params(p)
    p64, x64, t64 = p.astype(np.float64), x.astype(np.float64), t.astype(np.float64)
    ty, tg = TOL[prec]
    y = net.forward(x)
    yr, _, _ = mlp.forward(p64, widths, x64)
    assert np.max(np.abs(y - yr)) <= ty * max(1.0, np.max(np.abs(yr)))
    loss, g = net.gradients(x, t)
    lr, gr = mlp.loss_and_grad(p64, widths, x64, t64)
    assert abs(loss - lr) <= ty * max(1.0, lr)
    assert np.max(np.abs(g - gr)) <= tg * max(1e-3, np.max(np.abs(gr)))
    net.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("batch", [1, 130, 1024])
def test_gathered_rows_equal_plain_rows(kd, prec, batch):
    """Rows selected by index in the products' loaders give the update of the same rows laid
    out in memory, bit for bit; indices outside the sample range are rows of zeros."""
    import torch
    widths = [5, 96, 40, 4]
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((300, 5)).astype(np.float32)
    t = rng.standard_normal((300, 4)).astype(np.float32)
    idx = rng.integers(0, 300, batch).astype(np.int32)
    if batch > 1:
        idx[:2] = (-1, 300)
    ok = (idx >= 0) & (idx < 300)
    sel = np.clip(idx, 0, 299)
    xb = torch.from_numpy(np.where(ok[:, None], x[sel], 0).astype(np.float32)).cuda()
    tb = torch.from_numpy(np.where(ok[:, None], t[sel], 0).astype(np.float32)).cuda()
    xd, td, idev = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), torch.from_numpy(idx).cuda()
    loss = torch.zeros(2, device="cuda")
    got = []
    for gather in (True, False):
        net = kd.MLP(widths)
        net.set_precision(kd.KD_MLP_BF16 if prec == "bf16" else kd.KD_MLP_FP32)
        net.set_params(mlp.init_params(widths, 4))
        for _ in range(3):
            if gather:
                net.train_step_gather(xd.data_ptr(), td.data_ptr(), 300, idev.data_ptr(), batch, 1e-3,
                                      loss_dev=loss[0].data_ptr())
            else:
                net.train_step(xb.data_ptr(), tb.data_ptr(), batch, 1e-3, loss_dev=loss[1].data_ptr())
        torch.cuda.synchronize()
        got.append(net.get_params())
        net.close()
    assert np.array_equal(got[0], got[1])
    assert float(loss[0]) == float(loss[1])


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("widths,batch", [
    ([264, 130, 36], 32), ([264, 130, 36], 200), ([128, 256, 8], 256), ([131, 67, 3], 129), ([20, 36, 4], 17)])
def test_wide_gathered_rows_equal_plain_rows(kd, prec, widths, batch):
    """Inputs wide enough for the loaders' vector loads: whole tiles, tiles cut off by the batch
    or the width, and rows whose stride forbids 16-byte loads, gathered (an index out of range
    included) and plain, bit for bit; the plain step's loss against the FP64 oracle."""
    import torch
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((300, widths[0])).astype(np.float32)
    t = rng.standard_normal((300, widths[-1])).astype(np.float32)
    idx = rng.integers(0, 300, batch).astype(np.int32)
    idx[:2] = (300, -1)
    ok = (idx >= 0) & (idx < 300)
    sel = np.clip(idx, 0, 299)
    xb = np.where(ok[:, None], x[sel], 0).astype(np.float32)
    tb = np.where(ok[:, None], t[sel], 0).astype(np.float32)
    p = mlp.init_params(widths, 4)
    xd, td, idev, xbd, tbd = (torch.from_numpy(a).cuda() for a in (x, t, idx, xb, tb))
    loss = torch.zeros(2, device="cuda")
    got = []
    for gather in (True, False):
        net = kd.MLP(widths)
        net.set_precision(kd.KD_MLP_BF16 if prec == "bf16" else kd.KD_MLP_FP32)
        net.set_params(p)
        if gather:
            net.train_step_gather(xd.data_ptr(), td.data_ptr(), 300, idev.data_ptr(), batch, 1e-3,
                                  loss_dev=loss[0:].data_ptr())
        else:
            net.train_step(xbd.data_ptr(), tbd.data_ptr(), batch, 1e-3, loss_dev=loss[1:].data_ptr())
        torch.cuda.synchronize()
        got.append(net.get_params())
        net.close()
    assert np.array_equal(got[0], got[1])
    assert float(loss[0]) == float(loss[1])
    want, _ = mlp.loss_and_grad(p.astype(np.float64), widths, xb.astype(np.float64), tb.astype(np.float64))
    assert abs(float(loss[1]) - want) <= TOL[prec][0] * max(1.0, want)
