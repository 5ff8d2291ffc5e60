"""Warm-start network kernels: BF16 tensor-core GEMM (all stride forms), the
network's gradients against the FP64 reference (tests/oracle), and training
that lowers the loss."""
import numpy as np
import pytest
import torch

from oracle import mlp_ref
from paper_2609_11923_gb300 import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(100, 70, 50), (64, 64, 32), (257, 129, 300), (1, 8, 176)])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True)])
def test_gemm_matches_bf16_rounded_fp64_products(m, n, k, ta, tb):
    rng = np.random.default_rng(m * 7 + n + k)
    A = rng.standard_normal((k, m) if ta else (m, k)).astype(np.float32)
    B = rng.standard_normal((n, k) if tb else (k, n)).astype(np.float32)
    bias = rng.standard_normal(n).astype(np.float32)
    Ad, Bd, bd = (torch.tensor(x, device="cuda") for x in (A, B, bias))
    C = torch.empty((m, n), dtype=torch.float32, device="cuda")
    sam, sak = (1, m) if ta else (k, 1)
    sbk, sbn = (1, k) if tb else (n, 1)
    s = int(torch.cuda.current_stream().cuda_stream)
    M._ck(M._lib.mlp_gemm(Ad.data_ptr(), 0, sam, sak, Bd.data_ptr(), 0, sbk, sbn, C.data_ptr(), None, n, m, n, k,
                          bd.data_ptr(), 1, 0, s))
    Aop = A.T if ta else A
    Bop = B.T if tb else B
    ref = np.maximum(mlp_ref.bf16_round(Aop) @ mlp_ref.bf16_round(Bop) + bias, 0.0)
    np.testing.assert_allclose(C.cpu().numpy(), ref, rtol=1e-4, atol=1e-4 * np.abs(ref).max())


def test_network_gradients_match_fp64_reference():
    rng = np.random.default_rng(0)
    B = 96
    X = rng.standard_normal((B, M.N_OUT * 22)).astype(np.float32)
    nact = rng.integers(1, M.N_OUT + 1, size=B).astype(np.int32)
    T = np.zeros((B, M.N_OUT), dtype=np.float32)
    for i in range(B):
        p = rng.random(nact[i])
        T[i, :nact[i]] = p / p.sum()
    net = M.MLP(X.shape[1], seed=3)
    loss = net.loss_and_grad(torch.tensor(X, device="cuda"), torch.tensor(nact, device="cuda"),
                             torch.tensor(T, device="cuda"))
    W, b = net.numpy_params()
    gW, gb = net.numpy_grads()
    rl, rW, rb = mlp_ref.loss_and_grads(W, b, X.astype(np.float64), nact, T.astype(np.float64), bf16=True)
    assert loss == pytest.approx(rl, rel=1e-4)
    # element by element: both sides round the same operands to BF16; what
    # is left is FP32 against FP64 accumulation and activations whose BF16
    # rounding flips on the last bit (2^-8 of one term), so each entry must
    # agree to 2% of itself or 0.5% of the tensor's largest entry
    for g, r in zip(gW + gb, rW + rb):
        np.testing.assert_allclose(g, r, rtol=2e-2, atol=5e-3 * np.abs(r).max())


def test_training_lowers_the_loss_on_a_fixed_task():
    rng = np.random.default_rng(1)
    n, F = 8192, M.N_OUT * 22
    X = rng.standard_normal((n, F)).astype(np.float32)
    Wt = rng.standard_normal((F, M.N_OUT)) * 0.5
    nact = np.full(n, 4, dtype=np.int32)
    z = X @ Wt
    z[:, 4:] = -np.inf
    T = np.exp(z - z.max(1, keepdims=True))
    T = (T / T.sum(1, keepdims=True)).astype(np.float32)
    from paper_2609_11923_gb300 import warmstart

    net = warmstart.train(np.pad(X, ((0, 0), (0, warmstart.F_IN - F))), nact, T, epochs=4, batch=1024, lr=3e-3)
    assert net.history[-1] < 0.6 * net.history[0]


def _batch(rows, dim, seed=0):
    rng = np.random.default_rng(seed * 1000003 + rows * 257 + dim)
    X = rng.standard_normal((rows, dim)).astype(np.float32)
    nact = rng.integers(1, M.N_OUT + 1, size=rows).astype(np.int32)
    T = rng.random((rows, M.N_OUT)).astype(np.float32) * (np.arange(M.N_OUT) < nact[:, None])
    return X, nact, T / T.sum(1, keepdims=True)


# Fused network at the edges of its tiles (128 rows), operand groups (64
# rows), row splits and input blocks (64 features), against the FP64 reference
# with BF16-rounded operands; the bounds are those of the layer-by-layer test
# above (activations whose BF16 rounding flips on the last bit, 2^-8 of a term).
@pytest.mark.parametrize("dim", [4, 60, 64, 192, 196, 256])
@pytest.mark.parametrize("rows", [1, 63, 127, 128, 129, 2049])
def test_fused_network_matches_fp64_reference(rows, dim):
    X, nact, T = _batch(rows, dim)
    weight = np.random.default_rng(rows).random(rows).astype(np.float32) + 0.5
    net = M.MLP(dim, seed=3)
    assert net.fused
    for b in net.b:
        b.copy_(torch.randn(b.shape, generator=torch.Generator(device="cuda").manual_seed(dim), device="cuda"))
    put = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    W, b = net.numpy_params()
    z = mlp_ref.forward(W, b, X.astype(np.float64), bf16=True)[-1]
    z = np.where(np.arange(M.N_OUT) < nact[:, None], z, -np.inf)
    p = np.exp(z - z.max(1, keepdims=True))
    p /= p.sum(1, keepdims=True)
    got = net.predict(put(X), put(nact)).cpu().numpy()
    np.testing.assert_allclose(got, p, rtol=0, atol=2e-2)
    np.testing.assert_array_equal(got[np.arange(M.N_OUT) >= nact[:, None]], 0.0)
    for w in (None, weight):
        loss = net.loss_and_grad(put(X), put(nact), put(T), None if w is None else put(w))
        rl, rW, rb = mlp_ref.loss_and_grads(W, b, X.astype(np.float64), nact, T.astype(np.float64),
                                            None if w is None else w.astype(np.float64), bf16=True)
        assert loss == pytest.approx(rl, rel=1e-3)
        gW, gb = net.numpy_grads()
        for g, r in zip(gW + gb, rW + rb):
            np.testing.assert_allclose(g, r, rtol=2e-2, atol=(5e-3 if rows > 128 else 2e-2) * np.abs(r).max())


def test_fused_network_takes_unaligned_rows_and_keeps_the_activations_available():
    X, nact, T = _batch(300, 192, seed=1)
    net = M.MLP(192, seed=5)
    base = torch.zeros(300 * 192 + 1, device="cuda")
    view = base[1:].view(300, 192)  # 4-byte aligned only
    view.copy_(torch.tensor(X))
    n = torch.tensor(nact, device="cuda")
    a, b = net.predict(view, n), net.predict(torch.tensor(X, device="cuda"), n)
    assert torch.equal(a, b)
    acts = net.acts
    assert len(acts) == 5 and acts[0].data_ptr() != 0 and torch.equal(acts[0].cpu(), torch.tensor(X))
    assert torch.allclose(torch.softmax(acts[-1].masked_fill(
        torch.arange(8, device="cuda") >= n[:, None], -torch.inf), 1), a, atol=1e-2)


def test_adam_steps_agree_between_the_fused_and_the_layer_by_layer_network():
    X, nact, T = (torch.tensor(x, device="cuda") for x in _batch(500, 192, seed=2))
    a, b = M.MLP(192, seed=7), M.MLP(192, seed=7)
    b.fused = False
    for _ in range(3):
        la, lb = a.loss_and_grad(X, nact, T), b.loss_and_grad(X, nact, T)
        assert la == pytest.approx(lb, rel=1e-4)
        for x, y in zip(a.gW + a.gb, b.gW + b.gb):  # the same gradients into both updates
            y.copy_(x)
        a.adam_step(1e-3)
        b.adam_step(1e-3)
        for x, y in zip(a.W + a.b + a.Wb + a.mW + a.vW, b.W + b.b + b.Wb + b.mW + b.vW):
            assert torch.equal(x, y)  # one formula, one rounding


def test_other_shapes_run_layer_by_layer():
    X, nact, T = _batch(70, 20, seed=4)
    net = M.MLP(20, hidden=(32, 48), seed=1)
    assert not net.fused
    loss = net.loss_and_grad(*(torch.tensor(x, device="cuda") for x in (X, nact, T)))
    W, b = net.numpy_params()
    rl, _, _ = mlp_ref.loss_and_grads(W, b, X.astype(np.float64), nact, T.astype(np.float64), bf16=True)
    assert loss == pytest.approx(rl, rel=1e-3)


def test_a_failed_inference_is_raised_by_check_and_by_the_next_pass():
    X, nact, T = (torch.tensor(x, device="cuda") for x in _batch(200, 192, seed=6))
    net = M.MLP(192, seed=1)
    p = net.predict(X, nact)
    net.check()
    for call in (net.check, lambda: net.predict(X, nact), lambda: net.loss_and_grad(X, nact, T)):
        net._err.fill_(1)  # what a kernel writes whose wait gave up
        with pytest.raises(RuntimeError, match="gave up"):
            call()
        net.check()
    assert torch.equal(net.predict(X, nact), p)


def test_activations_after_a_step_are_not_those_of_other_weights():
    X, nact, T = (torch.tensor(x, device="cuda") for x in _batch(200, 192, seed=8))
    net = M.MLP(192, seed=2)
    net.loss_and_grad(X, nact, T)
    first = [x.clone() for x in net.acts]
    net.loss_and_grad(X, nact, T)
    net.adam_step(1e-2)
    with pytest.raises(RuntimeError, match="gone"):
        net.acts
    net.predict(X, nact)
    X.mul_(2.0)
    with pytest.raises(RuntimeError, match="gone"):
        net.backward(torch.zeros(200, 8, device="cuda"))
    net.forward(X)
    assert not torch.equal(net.acts[1], first[1])


def test_gradients_in_one_flat_buffer_take_the_layer_by_layer_route():
    # views that are 4-byte aligned only, as a flat gradient buffer gives them
    X, nact, T = (torch.tensor(x, device="cuda") for x in _batch(300, 192, seed=9))
    a, b = M.MLP(192, seed=3), M.MLP(192, seed=3)
    flat = torch.zeros(1 + sum(g.numel() for g in a.gW), device="cuda")
    at, views = 1, []
    for g in a.gW:
        views.append(flat[at:at + g.numel()].view_as(g))
        at += g.numel()
    a.gW = views
    b.fused = False
    assert a.loss_and_grad(X, nact, T) == b.loss_and_grad(X, nact, T)
    for x, y in zip(a.gW + a.gb, b.gW + b.gb):
        assert torch.equal(x, y)


def test_a_write_into_the_bf16_weights_reaches_every_pass():
    X, nact, T = (torch.tensor(x, device="cuda") for x in _batch(300, 192, seed=10))
    a, b = M.MLP(192, seed=3), M.MLP(192, seed=3)
    b.fused = False
    for net in (a, b):
        net.Wb[1].mul_(0.5)
    assert torch.equal(a.predict(X, nact), b.predict(X, nact))
    assert a.loss_and_grad(X, nact, T) == b.loss_and_grad(X, nact, T)
    a.sync_bf16()
    assert a._packed() and torch.equal(a.Wb[1], a.W[1].bfloat16())
