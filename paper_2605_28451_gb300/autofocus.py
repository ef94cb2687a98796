"""Differentiable entropy autofocus: a torch.autograd.Function over the C ABI.

Forward computes the image entropy E(phi) of the azimuth-compressed,
phase-corrected data.  When a gradient will be asked for it also keeps the
FP32 image (up to KEEP_BYTES) for backward, which then runs the hand-written
adjoint alone: four transforms per range bin for a step instead of eight.
Without the image (evaluation only, larger scenes, no memory for it, the
tensor-core mode, saved-tensor hooks, rc or ha written in between) backward
calls ``sar_autofocus_grad``, which computes it again.  A write is seen by the
tensors' version counters: torch's own operations and this package's calls
advance them.  Where something else writes rc or ha (another library's kernel,
a replayed CUDA graph, a call given a bare address), it must advance them too
(``torch.autograd.graph.increment_version``) or wait until backward has run.
Only argument marshalling happens here.
"""

from __future__ import annotations

import torch
from torch.autograd import forward_ad

from . import bfpfft as B


class Workspace:
    """Device scratch for the autofocus calls at one azimuth length, and the
    arithmetic they run in (BFPFFT_ARITH_F32, or ARITH_F16_MUL_F32_ACC for the
    tensor-core transforms at n_az = 4096)."""

    def __init__(self, n_az: int, device, arith: int = B.ARITH_F32):
        self.arith = arith
        self.bytes = B.sar_autofocus_workspace_bytes(n_az)
        if self.bytes == 0:
            raise ValueError(f"unsupported azimuth length {n_az}")
        self.buf = torch.empty(self.bytes, dtype=torch.uint8, device=device)
        self.stats = torch.empty(4, dtype=torch.float64, device=device)


KEEP_BYTES = 512 << 20   # largest state kept between forward and backward


def _versions(rc, ha):
    """The tensors' version counters, or None where one has none to tell a change
    by (made under inference_mode, or not torch's)."""
    try:
        return rc._version, ha._version
    except (RuntimeError, AttributeError):
        return None


# The saved-tensor hooks in force, if any (offloading, compression,
# checkpointing).  Those are meant for saved inputs: the image, computed again in
# a fraction of the time that moving it takes, is not handed to them.
_saved_tensor_hooks = getattr(torch._C._autograd, "_top_saved_tensors_default_hooks", lambda ignore_tracing: None)


def _address(g):
    """The address of an upstream gradient if the value there is all there is to it,
    else None: it carries a graph or a tangent on, waits for a negation, or is a
    wrapper (a batch) without an address."""
    if torch.is_grad_enabled() or getattr(forward_ad, "_current_level", 0) >= 0 or type(g) is not torch.Tensor \
            or g.is_neg():
        return None
    try:
        return g.data_ptr()
    except RuntimeError:
        return None


class SarEntropy(torch.autograd.Function):
    """E = entropy(|A(rc . exp(-j phi))|^2); d E / d phi by the GPU adjoint.

    rc: device tensor [n_rg][n_az] in storage dtype rc_dtype (complex64 for
    BFPFFT_F32, float16 [n_rg][n_az][2] for BFPFFT_F16_BFP); ha: complex64
    [n_az]; phi: float32 [n_az] (requires grad).  Returns a float64 scalar.
    keep: backward will be asked for, so the image may be kept.
    """

    @staticmethod
    def forward(ctx, phi, rc, ha, rc_dtype: int, ws: Workspace, keep: bool = False):
        n_rg, n_az = rc.shape[0], rc.shape[1]
        phi_c = phi.detach()
        if not phi_c.is_contiguous():
            phi_c = phi_c.contiguous()
        ctx.rc, ctx.ha, ctx.rc_dtype, ctx.ws = rc, ha, rc_dtype, ws
        keep = keep and ws.arith == B.ARITH_F32 and n_rg > 0 and _saved_tensor_hooks(False) is None
        versions = _versions(rc, ha) if keep else None
        if versions is not None:
            size = B.sar_autofocus_state_bytes(n_az, n_rg)
            if 0 < size <= KEEP_BYTES:
                try:
                    state = torch.empty(size, dtype=torch.uint8, device=phi_c.device)
                except torch.cuda.OutOfMemoryError:
                    state = None
                if state is not None:
                    e = torch.empty((), dtype=torch.float64, device=phi_c.device)
                    # Addresses of what nobody else holds: no version counters to advance.
                    B.sar_autofocus_entropy_keep(rc, rc_dtype, phi_c, ha, n_az, n_rg, ws.stats, e.data_ptr(),
                                                 state.data_ptr(), size, ws.buf, ws.bytes)
                    ctx.save_for_backward(phi_c, state)
                    ctx.versions = versions
                    return e
        B.sar_autofocus_entropy(rc, rc_dtype, phi_c, ha, n_az, n_rg, ws.stats, ws.buf, ws.bytes, arith=ws.arith)
        ctx.save_for_backward(phi_c)
        return ws.stats[2].clone()

    @staticmethod
    def backward(ctx, g_e):
        phi_c, *kept = ctx.saved_tensors
        rc, ha, ws = ctx.rc, ctx.ha, ctx.ws
        n_rg, n_az = rc.shape[0], rc.shape[1]
        grad = torch.empty(n_az, dtype=torch.float32, device=phi_c.device)
        scale = None
        if kept and ws.arith == B.ARITH_F32 and ctx.versions == _versions(rc, ha):
            state = kept[0]
            # The library multiplies by g_e where that loses nothing: a product in
            # torch takes another 10 us of host time.
            scale = _address(g_e)
            B.sar_autofocus_grad_kept(rc, ctx.rc_dtype, phi_c, ha, n_az, n_rg, state, state.numel(), scale,
                                      grad.data_ptr(), ws.stats, ws.buf, ws.bytes)
        else:
            B.sar_autofocus_grad(rc, ctx.rc_dtype, phi_c, ha, n_az, n_rg, grad.data_ptr(), ws.stats, ws.buf, ws.bytes,
                                 arith=ws.arith)
        if scale is None:
            grad = g_e * grad            # g_e is a scalar: the product is FP32
        return grad, None, None, None, None, None


def entropy(phi, rc, ha, rc_dtype: int, ws: Workspace):
    return SarEntropy.apply(phi, rc, ha, rc_dtype, ws, phi.requires_grad and torch.is_grad_enabled())
