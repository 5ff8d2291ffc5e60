"""Warm-start network on the GPU: 3 hidden ReLU layers of 256, masked softmax
over at most 8 actions.

FP32 master weights with BF16 copies; every product (forward and both
backward products), the loss, the ReLU gradients, the bias gradients and the
Adam updates run in libcfr.so's kernels (include/mlp.h). PyTorch only holds
the device memory. Weight layout: W[l] is [fan_in, fan_out] row-major, so a
layer is h_out = relu(h_in @ W + b).
"""
from __future__ import annotations

import ctypes
import struct
from itertools import chain
from operator import is_, methodcaller
from typing import List, Optional

import numpy as np

from . import cfr

_lib = cfr._lib
_vp, _l, _i = ctypes.c_void_p, ctypes.c_long, ctypes.c_int
_lib.mlp_gemm.argtypes = [_vp, _i, _l, _l, _vp, _i, _l, _l, _vp, _vp, _l, _i, _i, _i, _vp, _i, _i, _vp]
_lib.mlp_softmax_xent.argtypes = [_vp, _i, _vp, _vp, _vp, _i, _vp, _vp, _vp, _vp]
_lib.mlp_relu_grad.argtypes = [_vp, _vp, _l, _vp]
_lib.mlp_colsum.argtypes = [_vp, _i, _i, _vp, _vp]
_lib.mlp_adam.argtypes = [_vp, _vp, _vp, _vp, _l, ctypes.c_float, ctypes.c_float, ctypes.c_float, ctypes.c_float, _l,
                          _vp, _vp]
_lib.mlp_to_bf16.argtypes = [_vp, _vp, _l, _vp]
_pp, _f32 = ctypes.POINTER(_vp), ctypes.c_float
_lib.mlp_net_predict.argtypes = [_vp, _i, _i, _vp, _pp, _vp, _vp, _vp, _vp]
_lib.mlp_net_grad.argtypes = [_vp, _i, _i, _vp, _pp, _vp, _vp, _vp, _pp, _pp, _vp, ctypes.c_size_t,
                              ctypes.POINTER(_vp), _vp]
_lib.mlp_net_adam.argtypes = [_pp, _pp, _pp, _pp, _pp, _vp, _i, _f32, _f32, _f32, _f32, _l, _vp]
for _f in ("mlp_net_predict", "mlp_net_grad", "mlp_net_adam"):
    getattr(_lib, _f).restype = ctypes.c_int
_lib.mlp_net_image_bytes.argtypes = [_i]
_lib.mlp_net_work_bytes.argtypes = [_i, _i]
_lib.mlp_net_image_bytes.restype = _lib.mlp_net_work_bytes.restype = ctypes.c_size_t
_lib.mlp_net_last_error.restype = ctypes.c_char_p
for _f in ("mlp_gemm", "mlp_softmax_xent", "mlp_relu_grad", "mlp_colsum", "mlp_adam", "mlp_to_bf16"):
    getattr(_lib, _f).restype = ctypes.c_int
_lib.mlp_last_error.restype = ctypes.c_char_p

N_OUT = 8
_DATA_PTR = methodcaller("data_ptr")


def _ck(rc):
    if rc != 0:
        raise RuntimeError("mlp: " + (_lib.mlp_last_error() or b"").decode())


def _net_ck(rc):
    if rc != 0:
        raise RuntimeError("mlp: " + (_lib.mlp_net_last_error() or b"").decode())


def _writes(t) -> int:
    """A tensor's write counter (an inference tensor has none: never written)."""
    try:
        return t._version
    except RuntimeError:
        return -1


def _p(t) -> int:
    return 0 if t is None else int(t.data_ptr())


_ARRAYS = {}


def _ptrs(ts):
    """The tensors' addresses as a C array (kept by its contents: building one
    takes as long as a launch)."""
    at = tuple(map(_DATA_PTR, ts))
    a = _ARRAYS.get(at)
    if a is None:
        if len(_ARRAYS) >= 64:
            _ARRAYS.clear()
        a = _ARRAYS[at] = (_vp * len(at))(*at)
    return a


class MLP:
    def __init__(self, in_dim: int, hidden=(256, 256, 256), out: int = N_OUT, seed: int = 0, device="cuda"):
        import torch

        self.torch = torch
        self.dev = torch.device(device)
        self.dims = [in_dim] + list(hidden) + [out]
        rng = np.random.default_rng(seed)
        # the biases, and the BF16 weights, are views of one tensor each: the
        # write counter that a tensor shares with its views then tells at once
        # whether a caller has written into any of them (_packed, acts)
        shapes = list(zip(self.dims[:-1], self.dims[1:]))
        self._flat_b, self.b = self._views([(fo,) for _, fo in shapes], torch.float32)
        self._flat_wb, self.Wb = self._views(shapes, torch.bfloat16)
        self._own_b, self._own_wb = tuple(self.b), tuple(self.Wb)
        self.W = []
        for fi, fo in shapes:
            lim = np.sqrt(6.0 / fi)  # He-uniform for ReLU layers
            w = rng.uniform(-lim, lim, size=(fi, fo)).astype(np.float32)
            self.W.append(torch.tensor(w, device=self.dev))
        self.gW = [torch.zeros_like(w) for w in self.W]
        self.gb = [torch.zeros_like(b) for b in self.b]
        self.mW = [torch.zeros_like(w) for w in self.W]
        self.vW = [torch.zeros_like(w) for w in self.W]
        self.mb = [torch.zeros_like(b) for b in self.b]
        self.vb = [torch.zeros_like(b) for b in self.b]
        self.step_no = 0
        self._acts, self._fused_pass = None, None  # (batch, write counters) of the last pass if it was a fused one
        # networks of the warm start's shape run through the fused kernels
        # (mlp_net_*), from packed images of the weights; any other shape
        # runs layer by layer through mlp_gemm
        self.fused = (self.dims[1:] == [256, 256, 256, N_OUT] and self.dev.type == "cuda"
                      and _lib.mlp_net_image_bytes(in_dim) > 0)
        self.img = self.work = None
        if self.fused:
            self.img = torch.zeros(_lib.mlp_net_image_bytes(in_dim), dtype=torch.uint8, device=self.dev)
            # set to 1 by an inference kernel whose bounded wait gave up
            # (page-locked: the host reads it without a copy)
            self._err = torch.zeros(1, dtype=torch.int32).pin_memory()
            self._failed = ctypes.c_int32.from_address(self._err.data_ptr())
        self.sync_bf16()

    def _views(self, shapes, dtype):
        """Zeros of these shapes, 512 bytes aligned as tensors of their own
        would be, in one tensor: that tensor and its views."""
        at = [0]
        for s in shapes:
            at.append(at[-1] + (int(np.prod(s)) + 255) // 256 * 256)
        flat = self.torch.zeros(at[-1], dtype=dtype, device=self.dev)
        return flat, [flat[a:a + int(np.prod(s))].view(s) for a, s in zip(at, shapes)]

    def _s(self) -> int:
        return int(self.torch.cuda.current_stream(self.dev).cuda_stream)

    def _raise_if_failed(self):
        if self.fused and self._failed.value:
            self._failed.value = 0
            raise RuntimeError("mlp: a bounded wait of an inference kernel gave up; its probabilities are NaN")

    def check(self) -> None:
        """Waits for the current stream and raises if an inference on it
        failed (so does the next pass of the network, without waiting)."""
        if self.fused:
            self.torch.cuda.current_stream(self.dev).synchronize()
            self._raise_if_failed()

    @property
    def acts(self):
        """The input, every hidden layer's output and the logits of the last
        pass in FP32. The fused passes keep none: after one of them they are
        computed here, on first use, from its batch and the weights, and once
        either has changed (adam_step, sync_bf16, a write into the tensors,
        other tensors in their place) they are gone, which raises."""
        if self._acts is None and self._fused_pass is not None:
            X, x, b = self._fused_pass
            if X is None or x != _writes(X) or b != _writes(self._flat_b) or not self._own(self.b, self._own_b) or not self._packed():
                raise RuntimeError("mlp: the activations of the last fused pass are gone (its weights or its batch have "
                                   "changed since); run forward(X)")
            self.forward(X)
        return self._acts

    @acts.setter
    def acts(self, value):
        self._acts, self._fused_pass = value, None

    @staticmethod
    def _own(now, own) -> bool:
        return all(map(is_, now, own))

    def _ran_fused(self, X):
        self._acts, self._fused_pass = None, (X, _writes(X), _writes(self._flat_b))

    def _weights_change(self):  # by a kernel, past the counters: Wb and its images together
        self._packed_at = _writes(self._flat_wb) if self._own(self.Wb, self._own_wb) else None
        if self._fused_pass is not None:
            self._fused_pass = (None, 0, 0)

    def _packed(self) -> bool:
        """Whether the packed images are those of Wb. A caller's write into Wb
        reaches only the layer-by-layer passes, until sync_bf16 or a step writes
        both; with other tensors in Wb's place those passes run for good."""
        return _writes(self._flat_wb) == self._packed_at and self._own(self.Wb, self._own_wb)

    def sync_bf16(self):
        self._weights_change()
        if self.fused:
            _net_ck(_lib.mlp_net_adam(self._all(self.W, self.b), None, None, None, _ptrs(self.Wb), _p(self.img),
                                      self.dims[0], 0.0, 0.0, 0.0, 0.0, 0, self._s()))
            return
        for w, wb in zip(self.W, self.Wb):
            _ck(_lib.mlp_to_bf16(_p(w), _p(wb), w.numel(), self._s()))

    @staticmethod
    def _all(weights, biases):
        return _ptrs(chain.from_iterable(zip(weights, biases)))

    def _rows_ok(self, X) -> bool:
        return (self.fused and self._packed() and X.dtype == self.torch.float32 and X.dim() == 2 and X.shape[0] > 0
                and X.shape[1] == self.dims[0])

    # ---------------------------------------------------------------- passes
    def forward(self, X) -> "torch.Tensor":
        """X: [B, in_dim] FP32 on the device. Keeps the activations."""
        torch = self.torch
        self._raise_if_failed()
        B = X.shape[0]
        acts = self.acts = [X]
        h = X
        L = len(self.W)
        for l in range(L):
            fo = self.dims[l + 1]
            out = torch.empty((B, fo), dtype=torch.float32, device=self.dev)
            # A(m, k) = h[m, k]; B(k, n) = Wb[k, n]
            _ck(_lib.mlp_gemm(_p(h), 0, h.shape[1], 1, _p(self.Wb[l]), 1, fo, 1, _p(out), None, fo, B, fo,
                              self.dims[l], _p(self.b[l]), 1 if l < L - 1 else 0, 0, self._s()))
            acts.append(out)
            h = out
        return h

    def backward(self, dlogits) -> None:
        """Gradients of every weight and bias given d loss / d logits."""
        torch = self.torch
        B = dlogits.shape[0]
        d, acts = dlogits, self.acts
        for l in range(len(self.W) - 1, -1, -1):
            fi, fo = self.dims[l], self.dims[l + 1]
            h_in = acts[l]
            # gW = h_in^T d : A(m=i, k=b) = h_in[b, i]; B(k=b, n=j) = d[b, j]
            _ck(_lib.mlp_gemm(_p(h_in), 0, 1, fi, _p(d), 0, fo, 1, _p(self.gW[l]), None, fo, fi, fo, B, None, 0, 0,
                              self._s()))
            _ck(_lib.mlp_colsum(_p(d), B, fo, _p(self.gb[l]), self._s()))
            if l > 0:
                dh = torch.empty((B, fi), dtype=torch.float32, device=self.dev)
                # dh = d W^T : A(m=b, k=j) = d[b, j]; B(k=j, n=i) = Wb[i, j]
                _ck(_lib.mlp_gemm(_p(d), 0, fo, 1, _p(self.Wb[l]), 1, 1, fo, _p(dh), None, fi, B, fi, fo, None, 0, 0,
                                  self._s()))
                _ck(_lib.mlp_relu_grad(_p(dh), _p(h_in), dh.numel(), self._s()))
                d = dh

    def _fused_grad(self, X, B, nact, target, weight, loss) -> bool:
        """Launches the fused pass; False, and nothing launched, if its kernels
        cannot write the gradient tensors (views that are not 16-byte aligned)."""
        need = _lib.mlp_net_work_bytes(self.dims[0], B)
        if self.work is None or self.work.numel() < need:
            self.work = self.torch.empty(need, dtype=self.torch.uint8, device=self.dev)
        rc = _lib.mlp_net_grad(_p(X), self.dims[0], B, _p(self.img), _ptrs(self.b), _p(nact), _p(target), _p(weight),
                               _ptrs(self.gW), _ptrs(self.gb), _p(self.work), self.work.numel(), ctypes.byref(loss),
                               self._s())
        if rc != 0 and any(g.data_ptr() % 16 for g in self.gW):
            return False
        _net_ck(rc)
        return True

    def loss_and_grad(self, X, nact, target, weight=None) -> float:
        torch = self.torch
        self._raise_if_failed()
        B = X.shape[0]
        loss = _vp()
        if self._rows_ok(X) and self._fused_grad(X, B, nact, target, weight, loss):
            self._ran_fused(X)
            at = loss.value - self.work.data_ptr()
            total, failed = struct.unpack("=fi", self.work[at:at + 8].cpu().numpy().tobytes())
            if failed:
                raise RuntimeError("mlp: a bounded wait of the training kernels gave up")
            return total / B
        logits = self.forward(X)
        dlog = torch.empty_like(logits)
        rows = torch.empty(B, dtype=torch.float32, device=self.dev)
        _ck(_lib.mlp_softmax_xent(_p(logits), N_OUT, _p(nact), _p(target), _p(weight), B, None, _p(dlog), _p(rows),
                                  self._s()))
        self.backward(dlog)
        return float(rows.sum().item()) / B

    def adam_step(self, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8) -> None:
        self.step_no += 1
        self._weights_change()
        if self.fused:
            _net_ck(_lib.mlp_net_adam(self._all(self.W, self.b), self._all(self.gW, self.gb),
                                      self._all(self.mW, self.mb), self._all(self.vW, self.vb), _ptrs(self.Wb),
                                      _p(self.img), self.dims[0], lr, b1, b2, eps, self.step_no, self._s()))
            return
        for w, g, m, v, wb in zip(self.W, self.gW, self.mW, self.vW, self.Wb):
            _ck(_lib.mlp_adam(_p(w), _p(g), _p(m), _p(v), w.numel(), lr, b1, b2, eps, self.step_no, _p(wb), self._s()))
        for b, g, m, v in zip(self.b, self.gb, self.mb, self.vb):
            _ck(_lib.mlp_adam(_p(b), _p(g), _p(m), _p(v), b.numel(), lr, b1, b2, eps, self.step_no, None, self._s()))

    def predict(self, X, nact) -> "torch.Tensor":
        """Probabilities of the rows. Asynchronous: check() raises if the pass
        failed, once they are used on the host."""
        torch = self.torch
        self._raise_if_failed()
        if self._rows_ok(X):
            prob = torch.empty((X.shape[0], N_OUT), dtype=torch.float32, device=self.dev)
            _net_ck(_lib.mlp_net_predict(_p(X), self.dims[0], X.shape[0], _p(self.img), _ptrs(self.b), _p(nact),
                                         _p(prob), _p(self._err), self._s()))
            self._ran_fused(X)
            return prob
        logits = self.forward(X)
        prob = torch.empty_like(logits)
        _ck(_lib.mlp_softmax_xent(_p(logits), N_OUT, _p(nact), None, None, X.shape[0], _p(prob), None, None,
                                  self._s()))
        return prob

    # ------------------------------------------------------------ host copies
    def numpy_params(self):
        return ([w.cpu().numpy().astype(np.float64) for w in self.W],
                [b.cpu().numpy().astype(np.float64) for b in self.b])

    def numpy_grads(self):
        return ([g.cpu().numpy().astype(np.float64) for g in self.gW],
                [g.cpu().numpy().astype(np.float64) for g in self.gb])
