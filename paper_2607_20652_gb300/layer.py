"""The DPB as a PyTorch layer: autograd around the C-ABI calls.

Forward runs dpb_forward, i.e. dpb_encode then dpb_decode (the code and the
decode's r are kept for the backward); backward runs dpb_backward, the gradient with the
selected set held fixed. The layer has no trainable parameters: its dictionary is the
parity construction (§2.1). With ``ema`` set, the layer keeps live
standardisation tables (§2.2 "Score Standardization"): forward adds the
batch's moment sums (level 0 over every row, levels >= 1 over a 64-row
sub-sample) with the tables it selected with, and backward, once it has used
sigma, makes the EMA step (summed across data-parallel ranks first).

Every step runs in the library's kernels; this file only moves tensors.
"""
from __future__ import annotations

from typing import Optional

import torch

from . import dpb


class _DPBFunction(torch.autograd.Function):
    # x of any leading shape: the rows are taken here, outside the graph, so
    # that no reshape node runs in the backward. y is allocated in x's shape and
    # written through its rows: the output must not be a view made in here, for
    # autograd refuses in-place work on such a view (layer(x).add_(x)).
    @staticmethod
    def forward(ctx, x, layer):
        rows = x.reshape(-1, layer.d).contiguous()
        T = rows.shape[0]
        ws = layer._workspace(T, x.device)
        stream = layer._stream(x.device)
        ev = layer._events("forward")
        r = torch.empty((T, layer.d), dtype=torch.float32, device=x.device)  # kept for the backward
        y = torch.empty(x.shape, dtype=rows.dtype, device=x.device)
        idx, val, _, _ = dpb.forward(layer.plan, rows, layer.mu, layer.sigma, workspace=ws, stream=stream, r_out=r,
                                     y=y.view(T, layer.d))
        if layer.ema is not None and layer.training:
            sample = dpb.sample_rows(T, layer.ema_rows, layer._gen, x.device)
            dpb.stats_accumulate(layer.plan, rows, sample, layer._acc, mu=layer.mu, sigma=layer.sigma, workspace=ws,
                                 stream=stream)
        if ev:
            ev[1].record()
        ctx.save_for_backward(rows, idx, val, r)
        ctx.layer = layer
        layer.__dict__["last_code"] = (idx, val)  # (a plain attribute: Module.__setattr__ looks for parameters)
        return y

    @staticmethod
    def backward(ctx, gy):
        rows, idx, val, r = ctx.saved_tensors
        layer = ctx.layer
        shape = gy.shape
        gy = gy.reshape(rows.shape).contiguous().to(rows.dtype)
        ws = layer._workspace(rows.shape[0], rows.device)
        stream = layer._stream(rows.device)
        ev = layer._events("backward")
        gx, gv = dpb.backward(layer.plan, rows, idx, val, gy, layer.sigma, workspace=ws, stream=stream, r=r)
        if layer.ema is not None and layer.training:
            dpb.ema_step(lambda a: None,
                         lambda a: dpb.stats_update(layer.plan, a, layer.ema, layer.mu, layer.sigma, stream=stream),
                         layer._acc, layer.group)
        if ev:
            ev[1].record()
        layer.__dict__["last_grad_val"] = gv
        return gx.view(shape), None


class _RawStream:
    """A stream handle with the one attribute the calls read."""
    __slots__ = ("cuda_stream",)

    def __init__(self, handle):
        self.cuda_stream = handle


class DPBLayer(torch.nn.Module):
    """y = decode(encode(x)) over the last dimension (d), bf16 rows.

    ``plan_kw`` are dpb.Plan's arguments (d, levels, m_bits, children, beam,
    k, ...). ``ema`` (the EMA weight alpha, or None) turns on live
    standardisation; ``ema_rows`` is the sub-sample size of levels >= 1.
    ``group`` is the data-parallel process group of the moment all-reduce.
    """

    def __init__(self, ema: Optional[float] = None, ema_rows: int = 64, seed: int = 0, group=None,
                 device=None, **plan_kw):
        super().__init__()
        plan_kw.setdefault("dtype", "bf16")
        self.plan = dpb.Plan(**plan_kw)
        self.d = self.plan.d
        self.ema, self.ema_rows, self.group = ema, ema_rows, group
        dev = torch.device(device or "cuda")
        self._acc = None
        if ema is not None:
            m = self.plan.n_features
            self.register_buffer("mu", torch.zeros(m, dtype=torch.float32, device=dev))
            self.register_buffer("sigma", torch.ones(m, dtype=torch.float32, device=dev))
            self._acc = dpb.stats_buffer(self.plan, dev)
            self._gen = torch.Generator().manual_seed(seed)
        else:
            self.register_buffer("mu", None)
            self.register_buffer("sigma", None)
        self._ws = None
        self.timing = None          # set to a list to collect (forward, backward) CUDA event pairs
        self.last_code = None
        self.last_grad_val = None

    def _workspace(self, T, device):
        n = self.plan._ws_bytes
        if self._ws is None or self._ws.numel() < n or self._ws.device != device:
            self._ws = torch.zeros(n, dtype=torch.uint8, device=device)
        return self._ws

    def _stream(self, device):
        if device.type != "cuda":
            raise ValueError(f"x must be on a CUDA device, not {device}")
        return _RawStream(dpb._raw_stream(device.index))

    def _events(self, which):
        if self.timing is None:
            return None
        ev = (torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
        ev[0].record(torch.cuda.current_stream())
        self.timing.append((which, ev))
        return ev

    def forward(self, x):
        if x.shape[-1] != self.d:
            raise ValueError(f"last dimension {x.shape[-1]} != d = {self.d}")
        return _DPBFunction.apply(x.to(self.plan.torch_dtype), self)
