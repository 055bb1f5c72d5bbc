"""Torch-facing wrapper of one EC-MoE layer context (argument marshalling only).

PyTorch supplies device memory and the current stream; every step of the layer runs in
libecmoe.so. Tensor layouts are those of include/ecmoe.h.
"""
from __future__ import annotations

import torch

from . import (EC_BF16, EC_F32, _check, ec_check_device, ec_ctx_create, ec_ctx_destroy,
               ec_ctx_profile, ec_ctx_set_capacity, ec_ctx_set_profiling, ec_ctx_set_residual,
               ec_ctx_set_shared, ec_ctx_set_tiles, ec_ctx_set_workspace, ec_kernel_launches,
               ec_rows_per_expert, ec_tc_capacity, ec_tc_ctx_create, ec_workspace_bytes, load)

_DT = {"f32": (EC_F32, torch.float32), "bf16": (EC_BF16, torch.bfloat16)}


def _stream(stream):
    """Handle of `stream`, or of the current device's current stream (asked for without making
    a Stream object: 2.8 us of a call's host time)."""
    if stream is not None:
        return stream.cuda_stream
    return torch._C._cuda_getCurrentRawStream(torch.cuda.current_device())


class ECMoELayer:
    """One layer shape: N tokens in groups `group_off`, E experts, capacities k_g."""

    def __init__(self, N, d, E, d_ff, group_off, k_g, dtype="bf16", device="cuda",
                 d_ff_shared=0):
        self.N, self.d, self.E, self.d_ff = int(N), int(d), int(E), int(d_ff)
        self.G = len(group_off) - 1
        self.code, self.tdtype = _DT[dtype]
        self.device = torch.device(device)
        self.d_ff_shared = int(d_ff_shared)
        self.ctx = ec_ctx_create(self.N, self.d, self.E, self.d_ff, self.G, group_off, k_g,
                                 self.code)
        if self.d_ff_shared:
            ec_ctx_set_shared(self.ctx, self.d_ff_shared)
        self.ws_bytes = ec_workspace_bytes(self.ctx)
        self.ws = torch.empty(self.ws_bytes, dtype=torch.uint8, device=self.device)
        ec_ctx_set_workspace(self.ctx, self.ws.data_ptr(), self.ws_bytes)

    @property
    def M(self) -> int:
        return ec_rows_per_expert(self.ctx)

    def set_capacity(self, k_g):
        ec_ctx_set_capacity(self.ctx, k_g)

    def set_capacity_async(self, k_g_dev, stream=None):
        """k_g from an int32 device tensor [G] in stream order (sum must keep M)."""
        self._call(load().ec_ctx_set_capacity_async, (k_g_dev,), stream)

    def set_residual(self, on: bool):
        """Y = X + EC(X) and dX = dY + EC input gradient (stacked layers)."""
        ec_ctx_set_residual(self.ctx, on)

    def set_tiles(self, policy: int):
        """Expert-GEMM tile policy: EC_TILES_AUTO, EC_TILES_256 or EC_TILES_512."""
        ec_ctx_set_tiles(self.ctx, policy)

    def _call(self, fn, tensors, stream):
        """One C call: context, the tensors' addresses (None: NULL), the stream."""
        status = fn(self.ctx, *[None if t is None else t.data_ptr() for t in tensors],
                    _stream(stream))
        if status:
            _check(self.ctx, status)

    def _empty(self, *shape, dtype=None):
        return torch.empty(shape, dtype=dtype or self.tdtype, device=self.device)

    def _selection(self):
        """Empty idx [E][M], gate [E][M] and S [E][N]."""
        E, M, dev, f32 = self.E, self.M, self.device, torch.float32
        return (torch.empty((E, M), dtype=torch.int32, device=dev),
                torch.empty((E, M), dtype=f32, device=dev),
                torch.empty((E, self.N), dtype=f32, device=dev))

    def _grads(self, with_bias):
        d, E, F, dev, f32 = self.d, self.E, self.d_ff, self.device, torch.float32
        empty = torch.empty
        return {
            "dX": empty((self.N, d), dtype=self.tdtype, device=dev),
            "dWr": empty((d, E), dtype=f32, device=dev),
            "dbr": empty((E,), dtype=f32, device=dev) if with_bias else None,
            "dWg": empty((E, d, F), dtype=f32, device=dev),
            "dWu": empty((E, d, F), dtype=f32, device=dev),
            "dWd": empty((E, F, d), dtype=f32, device=dev),
        }

    def route(self, X=None, Wr=None, br=None, S_in=None, stream=None):
        """Selection only. Returns (idx [E][M] int32, gate [E][M] f32, S [E][N] f32)."""
        idx, gate, S = self._selection()
        self._call(load().ec_route, (X, Wr, br, S_in, S, idx, gate), stream)
        return idx, gate, S

    def forward(self, X, Wr, br, Wg, Wu, Wd, Y=None, stream=None, outputs=True, shared=None):
        """Y = EC-MoE(X) (+ shared experts). Returns (Y, idx, gate, S); idx/gate/S are None if
        outputs=False. shared = (Wg_s, Wu_s, Wd_s) in concatenated form when configured."""
        Y = self._empty(self.N, self.d) if Y is None else Y
        idx, gate, S = self._selection() if outputs else (None, None, None)
        lib = load()
        if self.d_ff_shared:
            Wgs, Wus, Wds = shared
            self._call(lib.ec_moe_forward_shared,
                       (X, Wr, br, Wg, Wu, Wd, Wgs, Wus, Wds, Y, idx, gate, S), stream)
        else:
            self._call(lib.ec_moe_forward, (X, Wr, br, Wg, Wu, Wd, Y, idx, gate, S), stream)
        # the backward pass reads these through the pointers the context remembered
        self._keep = (X, Wr, br, Wg, Wu, Wd, shared)
        return Y, idx, gate, S

    def backward(self, dY, grads=None, stream=None, with_bias=False):
        """Gradients of <dY, Y> for the last forward. Returns a dict of tensors."""
        g = grads or self._grads(with_bias)
        main = (dY, g["dX"], g["dWr"], g.get("dbr"), g["dWg"], g["dWu"], g["dWd"])
        if self.d_ff_shared:
            for k, shape in (("dWg_s", (self.d, self.d_ff_shared)),
                             ("dWu_s", (self.d, self.d_ff_shared)),
                             ("dWd_s", (self.d_ff_shared, self.d))):
                if g.get(k) is None:
                    g[k] = self._empty(*shape, dtype=torch.float32)
            self._call(load().ec_moe_backward_shared,
                       main + (g["dWg_s"], g["dWu_s"], g["dWd_s"]), stream)
        else:
            self._call(load().ec_moe_backward, main, stream)
        return g

    def set_profiling(self, on: bool):
        ec_ctx_set_profiling(self.ctx, on)

    def profile(self):
        """[(kernel, ms)] of every launch since profiling was switched on."""
        return ec_ctx_profile(self.ctx)

    @property
    def launches(self) -> int:
        return ec_kernel_launches(self.ctx)

    def check(self, stream=None):
        """Synchronise and raise if a kernel reported a device-side timeout."""
        ec_check_device(self.ctx, _stream(stream))

    def close(self):
        if self.ctx is not None:
            ec_ctx_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def tc_capacity(cf, k, N, E) -> int:
    """Token-choice expert capacity for a capacity factor (computed by the library's
    ec_tc_capacity); -1 (no cap, dropless) when cf is None or <= 0."""
    return ec_tc_capacity(cf, k, N, E)


class TCMoELayer(ECMoELayer):
    """Token-choice layer of the same shape (bf16): every token takes its k best experts,
    each expert keeps at most `capacity` tokens (-1: dropless)."""

    def __init__(self, N, d, E, d_ff, k, capacity=-1, dtype="bf16", device="cuda"):
        self.N, self.d, self.E, self.d_ff = int(N), int(d), int(E), int(d_ff)
        self.k, self.capacity = int(k), int(capacity)
        self.G = 1
        self.code, self.tdtype = _DT[dtype]
        self.device = torch.device(device)
        self.d_ff_shared = 0
        self.ctx = None
        self.ctx = ec_tc_ctx_create(self.N, self.d, self.E, self.d_ff, self.k, self.capacity,
                                    self.code)
        self.ws_bytes = ec_workspace_bytes(self.ctx)
        self.ws = torch.empty(self.ws_bytes, dtype=torch.uint8, device=self.device)
        ec_ctx_set_workspace(self.ctx, self.ws.data_ptr(), self.ws_bytes)

    def route(self, *a, **kw):
        raise NotImplementedError("token choice routes inside forward()")

    def forward(self, X, Wr, br, Wg, Wu, Wd, Y=None, stream=None, outputs=True, shared=None):
        """Y = TC-MoE(X). Returns (Y, choice [N][k], gate [N][k], kept [N][k], load [E],
        S [N][E]); all but Y are None if outputs=False."""
        if shared is not None:
            raise ValueError("token-choice layers have no shared experts")
        Y = self._empty(self.N, self.d) if Y is None else Y
        outs = [None] * 5
        if outputs:
            outs = [self._empty(self.N, self.k, dtype=torch.int32),
                    self._empty(self.N, self.k, dtype=torch.float32),
                    self._empty(self.N, self.k, dtype=torch.int32),
                    self._empty(self.E, dtype=torch.int32),
                    self._empty(self.N, self.E, dtype=torch.float32)]
        self._call(load().ec_tc_forward, (X, Wr, br, Wg, Wu, Wd, Y, *outs), stream)
        self._keep = (X, Wr, br, Wg, Wu, Wd)
        return (Y, *outs)

    def backward(self, dY, grads=None, stream=None, with_bias=False):
        g = grads or self._grads(with_bias)
        self._call(load().ec_tc_backward,
                   (dY, g["dX"], g["dWr"], g.get("dbr"), g["dWg"], g["dWu"], g["dWd"]), stream)
        return g
