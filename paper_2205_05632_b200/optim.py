"""COMP-AMS as the optimizer of a torch model: n workers = n micro-batches whose gradients are kept
apart, compressed separately with error feedback and averaged by the server (Algorithm 2).

The model's parameters are re-pointed at slices of one flat fp32 tensor theta, the vector Algorithm 2
updates; every parameter tensor is one block of the compressor ("the blocks are usually the layers",
Section 3.1) unless whole_vector is set. Per step:

    for i in range(n_workers):
        loss_i = ...            # forward / backward of worker i's micro-batch
        loss_i.backward()
        opt.collect(i)          # row i of G <- the gradients, which are then cleared
    opt.step()                  # one COMP-AMS iteration; the model's parameters move with theta

torch is used for the model and its autograd; the optimizer step itself runs in the CUDA library.
"""
from __future__ import annotations

import ctypes
from typing import Iterable, List

import numpy as np
import torch

from .binding import RANDK, TOPK, CompAMS, CompAMSError, _check, load_library


class CompAMSOptimizer:
    def __init__(self, params: Iterable[torch.nn.Parameter], n_workers: int, compressor: int = TOPK,
                 k_ratio: float = 0.01, whole_vector: bool = False, lr: float = 1e-3, beta1: float = 0.9,
                 beta2: float = 0.999, eps: float = 1e-8, seed: int = 0):
        self.params: List[torch.nn.Parameter] = [p for p in params if p.requires_grad]
        if not self.params:
            raise CompAMSError("no trainable parameters")
        dev = self.params[0].device
        if dev.type != "cuda" or any(p.device != dev or p.dtype != torch.float32 for p in self.params):
            raise CompAMSError("all parameters must be float32 tensors on one CUDA device")
        sizes = [p.numel() for p in self.params]
        self.offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        self.d = int(self.offsets[-1])
        self.n = int(n_workers)
        # theta: the flat parameter vector; the model's tensors become views of it
        self.theta = torch.empty(self.d, dtype=torch.float32, device=dev)
        for p, lo, hi in zip(self.params, self.offsets[:-1], self.offsets[1:]):
            self.theta[lo:hi].copy_(p.data.reshape(-1))
            p.data = self.theta[lo:hi].view(p.shape)
        self.G = torch.zeros(self.n, self.d, dtype=torch.float32, device=dev)
        # collect(): the tensors that have elements, their places in a row, and room for their gradients' addresses
        self._pieces = [(p, 4 * size) for p, size in zip(self.params, sizes) if size]
        places = [int(o) for o, size in zip(self.offsets, sizes) if size] + [self.d]
        self._places = (ctypes.c_int64 * len(places))(*places)
        self._addresses = (ctypes.c_void_p * len(self._pieces))()
        blocks = np.array([0, self.d], dtype=np.int64) if whole_vector else self.offsets
        with torch.cuda.device(dev):
            self.opt = CompAMS(self.n, self.d, blocks, compressor, k_ratio, lr, beta1, beta2, eps)
            if compressor == RANDK:
                self.opt.set_seed(seed)  # Random-k: the seed of the index sets

    def collect(self, worker: int) -> None:
        """Row `worker` of G <- the gradients accumulated since the last collect(); they are cleared."""
        if not 0 <= worker < self.n:
            raise CompAMSError("worker %d outside [0, %d)" % (worker, self.n))
        # one kernel for all tensors, which reads them by their addresses
        dev = self.G.device
        index = dev.index
        grads, addresses = [], []  # (the former keeps the packed copies until the kernel is enqueued)
        for p, nbytes in self._pieces:
            g = p.grad
            if g is not None:
                # not as the kernel reads it, after a model.half() or .cpu() for instance, channels-last, an expanded view; the
                # negative of what lies in memory (the imaginary part of a conjugate), which only one element can be and be packed
                if g.nbytes != nbytes or g.get_device() != index or not g.is_contiguous() or (nbytes == 4 and g.is_neg()):
                    if 4 * g.numel() != nbytes:
                        raise CompAMSError("a gradient of %d elements for a parameter of %d" % (g.numel(), nbytes // 4))
                    g = g.to(dev, torch.float32).resolve_neg().contiguous()
                grads.append(g)
            addresses.append(None if g is None else g.data_ptr())
        self._addresses[:] = addresses
        with torch.cuda.device(dev):
            stream = torch.cuda.current_stream(dev).cuda_stream
            _check(load_library().compams_collect(self.G.data_ptr() + 4 * self.d * worker, self._addresses, self._places,
                                                  len(addresses), stream), "compams_collect")
        for p in self.params:
            p.grad = None

    def step(self) -> None:
        self.opt.step(self.G, self.theta)

    def set_lr(self, lr: float) -> None:
        self.opt.set_lr(lr)

    def close(self) -> None:
        self.opt.close()
