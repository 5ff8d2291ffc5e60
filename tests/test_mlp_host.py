"""Host side of the network (no GPU): a failed inference is reported before its
probabilities are used."""
import numpy as np
import pytest
import torch

import gamegen as gg
from paper_2609_11923_gb300 import mlp, warmstart


def bare(err=0):
    """A network without its tensors, in the state that its fused passes leave."""
    net = mlp.MLP.__new__(mlp.MLP)
    net.torch, net.dev, net.fused = torch, torch.device("cpu"), True
    net._err = torch.tensor([err], dtype=torch.int32)
    net._acts, net._X = None, None
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
