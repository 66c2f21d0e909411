"""``torch.autograd.Function`` over the FP32 fitness kernels of libpsso.so
(psso_fitness_forward_ws / psso_fitness_backward_ws): f = fitness(X) for the
rows of a CUDA float32 tensor, differentiable with respect to X.  The rotated
functions' products z = M (x - o) and M^T df/dz run on the tensor cores, in a
workspace taken from torch's caching allocator.

The tensors are plumbing only: both passes run in the library's kernels, on
torch's current CUDA stream.
"""
from __future__ import annotations

import torch

from . import (FN, PSSO_ROT_ACKLEY, PSSO_ROT_ELLIPSOID, PSSO_ROT_RASTRIGIN,
               psso_fitness_backward_ws, psso_fitness_forward_ws, psso_fitness_workspace_size)


def _ptr(t):
    return None if t is None else t.data_ptr()


def _stream(device):
    return torch.cuda.current_stream(device).cuda_stream


try:  # the stream's handle without a torch.cuda.Stream object around it
    from torch._C import _cuda_getCurrentRawStream as _raw_stream
except ImportError:
    _raw_stream = None


def _workspace(fn, N, D, device):
    if fn not in _ROTATED:      # no call needed: the other functions use no workspace
        return None, 0
    n = psso_fitness_workspace_size(fn, N, D)
    if n == 0:
        return None, 0
    # the caching allocator returns blocks aligned to at least 512 bytes
    return torch.empty(n, dtype=torch.uint8, device=device), n


_ROTATED = (PSSO_ROT_ELLIPSOID, PSSO_ROT_RASTRIGIN, PSSO_ROT_ACKLEY)


def _data(t, device):
    """t as a contiguous float32 tensor on the device (itself if it is one)."""
    if t is None or (t.dtype is torch.float32 and t.device == device and t.is_contiguous()):
        return t
    return t.to(device, torch.float32).contiguous()


class Fitness(torch.autograd.Function):
    @staticmethod
    def forward(ctx, X, fn, shift, weights=None, rotation=None):
        if not (X.is_cuda and X.dtype is torch.float32 and X.dim() == 2):
            raise TypeError("X must be a 2-D float32 CUDA tensor")
        device = X.device
        X = X.contiguous()
        N, D = X.shape
        shift, weights, rotation = _data(shift, device), _data(weights, device), _data(rotation, device)
        f = torch.empty(N, device=device, dtype=torch.float32)
        fn = FN[fn] if isinstance(fn, str) else int(fn)
        ws, nws = _workspace(fn, N, D, device)
        stream = _raw_stream(device.index) if _raw_stream else _stream(device)
        psso_fitness_forward_ws(fn, N, D, X.data_ptr(), shift.data_ptr(), _ptr(weights),
                                _ptr(rotation), f.data_ptr(), _ptr(ws), nws, stream)
        ctx.save_for_backward(X, shift, weights, rotation)
        ctx.fn = fn
        return f

    @staticmethod
    def backward(ctx, grad_f):
        X, shift, weights, rotation = ctx.saved_tensors
        N, D = X.shape
        device = X.device
        grad_f = _data(grad_f, grad_f.device)
        gX = torch.empty_like(X)
        ws, nws = _workspace(ctx.fn, N, D, device)
        stream = _raw_stream(device.index) if _raw_stream else _stream(device)
        psso_fitness_backward_ws(ctx.fn, N, D, X.data_ptr(), shift.data_ptr(), _ptr(weights),
                                 _ptr(rotation), grad_f.data_ptr(), gX.data_ptr(), _ptr(ws), nws,
                                 stream)
        return gX, None, None, None, None


def fitness(X, fn, shift, weights=None, rotation=None):
    """Differentiable FP32 fitness of the rows of X (N x D, float32, CUDA)."""
    return Fitness.apply(X, fn, shift, weights, rotation)
