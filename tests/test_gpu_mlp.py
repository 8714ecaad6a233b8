"""The network's CUDA kernels against the FP64 reference."""
import numpy as np
import pytest

from oracle import mlp_ref as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1411_2181_gb300 import build
    build.build()
    from paper_1411_2181_gb300 import mlp
    return mlp


def batch(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(n, 6)).astype(np.float32)
    t = np.column_stack([rng.uniform(0, 0.5, n), rng.uniform(-0.5, 0.5, n), rng.integers(0, 2, n),
                         rng.uniform(0, 1, n)]).astype(np.float32)
    mask = (rng.uniform(size=n) > 0.2).astype(np.float32)
    return x, t, mask


def per_tensor_err(g, ref):
    errs = []
    for (gw, gb), (rw, rb) in zip(R.unpack(g.astype(np.float64)), R.unpack(ref)):
        for a, b in ((gw, rw), (gb, rb)):
            errs.append(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))
    return max(errs)


@pytest.mark.parametrize("B", [1, 37, 300])
def test_fp32_forward_and_gradient(M, B):
    net = M.MLP(max_batch=512, bf16=False)
    p = M.init_params(3)
    net.set_params(p)
    x, t, mask = batch(B, B)
    y = net.forward(x)
    yr = R.forward(p.astype(np.float64), x.astype(np.float64))
    assert np.abs(y - yr).max() / np.abs(yr).max() < 1e-5
    loss = net.loss_grad(x, t, mask)
    lr_, gr = R.loss_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64), mask)
    assert abs(loss - lr_) / abs(lr_) < 1e-5
    assert per_tensor_err(net.grads(), gr) < 1e-5


def test_bf16_weights_gradient(M):
    """BF16 weights: compare with the reference evaluated at the BF16-rounded
    weights; accumulation stays FP32."""
    import torch
    net = M.MLP(max_batch=512, bf16=True)
    p = M.init_params(4)
    net.set_params(p)
    pb = torch.tensor(p).to(torch.bfloat16).to(torch.float64).numpy()
    x, t, mask = batch(256, 9)
    net.loss_grad(x, t, mask)
    _, gr = R.loss_grad(pb, x.astype(np.float64), t.astype(np.float64), mask)
    assert per_tensor_err(net.grads(), gr) < 1e-2
    y = net.forward(x)
    yr = R.forward(pb, x.astype(np.float64))
    assert np.abs(y - yr).max() / np.abs(yr).max() < 1e-2


def test_adamw_steps_match_reference(M):
    net = M.MLP(max_batch=128, bf16=False)
    p = M.init_params(5)
    net.set_params(p)
    x, t, mask = batch(64, 11)
    pr = p.astype(np.float64)
    m = np.zeros_like(pr)
    v = np.zeros_like(pr)
    for step in range(1, 4):
        net.loss_grad(x, t, mask)
        g = net.grads().astype(np.float64)
        net.adamw(lr=1e-3, weight_decay=1e-2)
        pr, m, v = R.adamw(pr, m, v, g, step, lr=1e-3, wd=1e-2)
        assert np.abs(net.get_params() - pr).max() < 1e-6


def test_training_reduces_loss(M):
    rng = np.random.default_rng(0)
    x = rng.uniform(-1, 1, size=(1024, 6)).astype(np.float32)
    t = np.column_stack([0.3 * np.tanh(x[:, 0]), 0.2 * x[:, 1] * x[:, 2], (x[:, 0] + x[:, 3] > 0),
                         np.abs(x[:, 4])]).astype(np.float32)
    net = M.MLP(max_batch=1024, bf16=True)
    net.set_params(M.init_params(0))
    hist = net.fit(x, t, epochs=300, lr=3e-3, batch=256)
    assert hist[-1] < 0.25 * hist[0]


# a forward error of each of five layers of at most 128 FP32 roundings each,
# passed back through as many: 5 x 128 x 2^-24, relative to the largest entry
TOL_CHAIN = 5 * 128 * 2.0 ** -24


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("B", [2, 5, 63, 64, 65, 1025, 2432, 2449])
def test_row_blocks_and_batch_parts(M, B, bf16):
    """Batches at the edges of the row blocks (2, 4 and 16 rows) and of the
    weight gradient's parts (one, several, the most), with FP32 and BF16
    weights: outputs, loss and gradient against the reference evaluated at
    the weights the kernels read; repeated calls give the same bits."""
    import torch
    net = M.MLP(max_batch=2449, bf16=bf16)
    p = M.init_params(B)
    net.set_params(p)
    pr = p.astype(np.float64)
    if bf16:
        pr = torch.tensor(p).to(torch.bfloat16).to(torch.float64).numpy()
    x, t, mask = batch(B, B + 1)
    y = net.forward(x)
    yr = R.forward(pr, x.astype(np.float64))
    assert np.abs(y - yr).max() / np.abs(yr).max() < TOL_CHAIN
    loss = net.loss_grad(x, t, mask)
    g = net.grads()
    lr_, gr = R.loss_grad(pr, x.astype(np.float64), t.astype(np.float64), mask)
    assert abs(loss - lr_) / abs(lr_) < TOL_CHAIN
    assert per_tensor_err(g, gr) < TOL_CHAIN
    assert net.loss_grad(x, t, mask) == loss and np.array_equal(net.grads(), g)
    assert np.array_equal(net.forward(x), y)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n,bs", [(1, 1), (37, 37), (300, 64), (130, 65)])
def test_epoch_equals_single_steps(M, n, bs, bf16):
    """An epoch in one call gives the bits of its mini-batches one by one
    (gradient, then step): parameters, last gradient and loss."""
    import ctypes as ct
    import torch
    p = M.init_params(n)
    x, t, mask = batch(n, n + 2)
    a, b = M.MLP(max_batch=bs, bf16=bf16), M.MLP(max_batch=bs, bf16=bf16)
    a.set_params(p)
    b.set_params(p)
    d = [torch.from_numpy(v).cuda() for v in (x, t, mask)]
    torch.cuda.synchronize()
    for _ in range(2):
        tot = ct.c_double()
        assert M._lib.lbfe_mlp_epoch(a._h, *[ct.c_void_p(v.data_ptr()) for v in d], n, bs, 1e-3, 0.9, 0.999, 1e-8, 1e-2,
                                     ct.byref(tot)) == 0
        want = 0.0
        for s in range(0, n, bs):
            e = slice(s, s + bs)
            want += b.loss_grad(x[e], t[e], mask[e]) * len(x[e])
            b.adamw(lr=1e-3, weight_decay=1e-2)
        assert tot.value == want
        assert np.array_equal(a.get_params(), b.get_params()) and np.array_equal(a.grads(), b.grads())
    assert M._lib.lbfe_mlp_epoch(a._h, *[ct.c_void_p(v.data_ptr()) for v in d], n, bs + 1, 1e-3, 0.9, 0.999, 1e-8, 0.0,
                                 None) != 0


@pytest.mark.parametrize("B", [1, 37, 4096])
@pytest.mark.parametrize("off", [0, 4, 6, 20])
def test_outputs_over_the_inputs(M, B, off):
    """y may overlap x: the result is the one of separate buffers, wherever in
    x's rows it starts."""
    import ctypes as ct
    import torch
    net = M.MLP(max_batch=B)
    net.set_params(M.init_params(5))
    x = batch(B, 9)[0]
    buf = torch.zeros(6 * B + 4 * B + 32, device="cuda")
    want = torch.zeros(4 * B, device="cuda")
    for _ in range(3):
        buf[:6 * B] = torch.from_numpy(x.ravel())
        torch.cuda.synchronize()
        assert M._lib.lbfe_mlp_forward(net._h, ct.c_void_p(buf.data_ptr()), B, ct.c_void_p(want.data_ptr())) == 0
        assert M._lib.lbfe_mlp_forward(net._h, ct.c_void_p(buf.data_ptr()), B, ct.c_void_p(buf.data_ptr() + 4 * off)) == 0
        torch.cuda.synchronize()
        assert torch.equal(buf[off:off + 4 * B], want) and want.abs().max() > 0


def test_outputs_in_pinned_host_memory(M):
    """A buffer outside the device takes the copy's path: same bits."""
    import ctypes as ct
    import torch
    net = M.MLP(max_batch=341)
    net.set_params(M.init_params(5))
    x = torch.from_numpy(batch(341, 9)[0]).cuda()
    host, dev = torch.zeros(341, 4).pin_memory(), torch.zeros(341, 4, device="cuda")
    torch.cuda.synchronize()
    for y in (host, dev):
        assert M._lib.lbfe_mlp_forward(net._h, ct.c_void_p(x.data_ptr()), 341, ct.c_void_p(y.data_ptr())) == 0
    torch.cuda.synchronize()
    assert torch.equal(dev.cpu(), host)


@pytest.mark.parametrize("B", [4560, 4561, 4577, 8193])
def test_large_batches_of_fp32_weights(M, B):
    """At and beyond the batch where FP32 weights go layer by layer, also with
    the outputs over the inputs: against the reference."""
    import ctypes as ct
    import torch
    net = M.MLP(max_batch=B, bf16=False)
    p = M.init_params(3)
    net.set_params(p)
    x = batch(B, 4)[0]
    want = R.forward(p.astype(np.float64), x.astype(np.float64))
    y = net.forward(x)
    assert np.abs(y - want).max() / np.abs(want).max() < TOL_CHAIN
    buf = torch.from_numpy(x.ravel()).cuda()
    torch.cuda.synchronize()
    assert M._lib.lbfe_mlp_forward(net._h, ct.c_void_p(buf.data_ptr()), B, ct.c_void_p(buf.data_ptr())) == 0
    torch.cuda.synchronize()
    assert np.array_equal(buf[:4 * B].cpu().numpy().reshape(B, 4), y)
