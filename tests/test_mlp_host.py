"""Host side of the network (no GPU): a failed inference is reported before its
probabilities are used, activations are never those of another pass, and the C
entries refuse what their kernels cannot read."""
import ctypes

import pytest
import torch

import gamegen as gg
from paper_2609_11923_gb300 import mlp, warmstart


def bare(err=0):
    """A network without most of its tensors, in the state that its fused passes leave."""
    net = mlp.MLP.__new__(mlp.MLP)
    net.torch, net.dev, net.fused = torch, torch.device("cpu"), True
    net._err = torch.tensor([err], dtype=torch.int32)
    net._failed = ctypes.c_int32.from_address(net._err.data_ptr())
    net._flat_wb, net._flat_b = torch.zeros(5), torch.zeros(4)
    net.Wb, net.b = list(net._flat_wb.split([3, 2])), list(net._flat_b.split([1, 3]))
    net._own_wb, net._own_b = tuple(net.Wb), tuple(net.b)
    net.dims = [4, 2]
    net._acts, net._fused_pass = None, None
    net._weights_change()
    return net


@pytest.mark.parametrize("call", [lambda n, x: n.predict(x, None), lambda n, x: n.loss_and_grad(x, None, None),
                                  lambda n, x: n.forward(x)], ids=["predict", "loss_and_grad", "forward"])
def test_the_pass_after_a_failed_inference_raises_once(call):
    net = bare(err=1)
    with pytest.raises(RuntimeError, match="gave up"):
        call(net, torch.zeros(2, 4))
    assert int(net._err[0]) == 0
    net._raise_if_failed()


def test_warm_start_raises_on_a_failed_inference():
    g = gg.endgame(3, 1000)

    class Failing(mlp.MLP):
        def __init__(self):
            self.dev, self.checked = torch.device("cpu"), False

        def predict(self, X, nact):
            return torch.full((X.shape[0], mlp.N_OUT), float("nan"))

        def check(self):
            raise RuntimeError("gave up")

    with pytest.raises(RuntimeError, match="gave up"):
        warmstart.warm_regrets(Failing(), g, 8.0)


@pytest.mark.parametrize("change", [lambda n, x: n._weights_change(), lambda n, x: x.add_(1.0), lambda n, x: n.b[0].zero_(),
                                    lambda n, x: n.b.__setitem__(1, torch.zeros(3)), lambda n, x: n.Wb[1].zero_()],
                         ids=["step", "batch", "bias", "other bias", "weights"])
def test_activations_of_a_fused_pass_are_gone_once_its_inputs_change(change):
    net, X = bare(), torch.zeros(2, 4)
    ran = []

    def forward(x):
        ran.append(x)
        net.acts = [x]

    net.forward = forward
    net._ran_fused(X)
    assert net.acts[0] is X and ran == [X]  # nothing has changed: computed on first use
    net._ran_fused(X)
    change(net, X)
    with pytest.raises(RuntimeError, match="gone"):
        net.acts
    forward(X)  # a layer-by-layer pass keeps its own
    net._weights_change()
    assert net.acts[0] is X


@pytest.mark.parametrize("change", [lambda n: n.Wb[1].add_(1.0), lambda n: n.Wb.__setitem__(0, torch.zeros(3))],
                         ids=["write", "replace"])
def test_changed_bf16_weights_leave_the_packed_images(change):
    net, X = bare(), torch.zeros(2, 4)
    assert net._rows_ok(X)
    net.b[0].add_(1.0)  # biases are read as they are
    assert net._rows_ok(X)
    change(net)
    assert not net._rows_ok(X)
    net._weights_change()  # what sync_bf16 and a step do as they write both
    assert net._rows_ok(X) == (net.Wb[0] is net._own_wb[0])


# addresses that are only looked at: every refusal comes before any launch
AT = 1 << 20


def ptrs(*at):
    return (ctypes.c_void_p * 4)(*at)


@pytest.mark.parametrize("img,prob", [(AT + 2, AT), (AT + 8, AT), (AT, AT + 4)])
def test_inference_refuses_misaligned_buffers(img, prob):
    rc = mlp._lib.mlp_net_predict(AT, 64, 5, img, ptrs(AT, AT, AT, AT), AT, prob, AT, None)
    assert rc == -1 and b"aligned" in mlp._lib.mlp_net_last_error()


@pytest.mark.parametrize("bad", ["img", "work", 0, 1, 2, 3])
def test_training_refuses_misaligned_buffers(bad):
    at = {k: AT + 4 * (k == bad) for k in ("img", "work", 0, 1, 2, 3)}
    loss = ctypes.c_void_p()
    rc = mlp._lib.mlp_net_grad(AT, 64, 5, at["img"], ptrs(AT, AT, AT, AT), AT, AT, None, ptrs(at[0], at[1], at[2], at[3]),
                               ptrs(AT, AT, AT, AT), at["work"], 1 << 40, ctypes.byref(loss), None)
    assert rc == -1 and b"aligned" in mlp._lib.mlp_net_last_error()
