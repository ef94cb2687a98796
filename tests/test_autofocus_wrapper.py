"""What the autofocus wrapper does around the library calls, with those replaced by a stand-in on the CPU whose entropy
is linear, E = sum c phi with c = sum over the range bins of rc: the gradient is c times the upstream gradient exactly."""

import ctypes

import pytest
import torch

from paper_2605_28451_gb300 import autofocus as GA
from paper_2605_28451_gb300 import bfpfft as B

N_AZ, N_RG = 8, 3


def column_sums(rc):
    return rc.sum(0)


def floats(address, count, ctype=ctypes.c_float):
    """The numbers at an address the wrapper handed over (the library never sees the tensors themselves)."""
    address = address if isinstance(address, int) else address.data_ptr()
    return torch.frombuffer((ctype * count).from_address(address), dtype=torch.float32 if ctype is ctypes.c_float
                            else torch.float64)


class Library:
    """The calls SarEntropy makes, and which of them were made."""

    def __init__(self, monkeypatch):
        self.calls = []
        monkeypatch.setattr(B, "sar_autofocus_workspace_bytes", lambda n_az: 64)
        monkeypatch.setattr(B, "sar_autofocus_state_bytes", lambda n_az, n_rg: 256 + 8 * n_az)
        for name in ("entropy", "entropy_keep", "grad", "grad_kept"):
            monkeypatch.setattr(B, "sar_autofocus_" + name, getattr(self, name))

    def entropy(self, rc, rc_dtype, phi, ha, n_az, n_rg, stats, ws, ws_bytes, arith=B.ARITH_F32, stream=None):
        self.calls.append("entropy")
        stats[2] = (column_sums(rc) * phi).sum()

    def entropy_keep(self, rc, rc_dtype, phi, ha, n_az, n_rg, stats, e, state, state_bytes, ws, ws_bytes, stream=None):
        self.calls.append("entropy_keep")
        floats(e, 1, ctypes.c_double).copy_((column_sums(rc) * phi).sum())
        floats(state, n_az).copy_(column_sums(rc))

    def grad(self, rc, rc_dtype, phi, ha, n_az, n_rg, grad, stats, ws, ws_bytes, arith=B.ARITH_F32, stream=None):
        self.calls.append("grad")
        floats(grad, n_az).copy_(column_sums(rc))

    def grad_kept(self, rc, rc_dtype, phi, ha, n_az, n_rg, state, state_bytes, scale, grad, stats, ws, ws_bytes,
                  stream=None):
        self.calls.append("grad_kept")
        floats(grad, n_az).copy_(floats(state, n_az))
        if scale is not None:
            floats(grad, n_az).mul_(floats(scale, 1, ctypes.c_double).item())


@pytest.fixture
def library(monkeypatch):
    return Library(monkeypatch)


def scene(seed=0):
    g = torch.Generator().manual_seed(seed)
    rc = torch.randint(-4, 5, (N_RG, N_AZ), generator=g).float()
    phi = torch.randint(-4, 5, (N_AZ,), generator=g).float().requires_grad_(True)
    return rc, torch.ones(N_AZ), phi, GA.Workspace(N_AZ, "cpu")


def test_gradient_stays_differentiable_in_the_upstream_gradient(library):
    rc, ha, phi, ws = scene()
    w = torch.tensor(3.0, dtype=torch.float64, requires_grad=True)
    grad, = torch.autograd.grad(w * GA.entropy(phi, rc, ha, B.F32, ws), phi, create_graph=True)
    assert library.calls == ["entropy_keep", "grad_kept"]
    assert grad.dtype == torch.float32 and torch.equal(grad, 3.0 * column_sums(rc))
    dw, = torch.autograd.grad(grad.sum(), w)
    assert dw == column_sums(rc).sum()


def test_directional_derivative(library):
    rc, ha, phi, ws = scene(1)
    v = torch.arange(1.0, N_AZ + 1)
    _, d = torch.autograd.functional.jvp(lambda p: GA.entropy(p, rc, ha, B.F32, ws), phi.detach(), v)
    assert d == (column_sums(rc) * v).sum()


def test_batched_upstream_gradients(library):
    rc, ha, phi, ws = scene(2)
    e = GA.entropy(phi, rc, ha, B.F32, ws)
    up = torch.tensor([1.0, -2.0, 5.0], dtype=torch.float64)
    grad, = torch.autograd.grad(e, phi, grad_outputs=up, is_grads_batched=True)
    assert grad.dtype == torch.float32 and torch.equal(grad, up.float()[:, None] * column_sums(rc))


def test_tangent_of_the_upstream_gradient(library):
    rc, ha, phi, ws = scene(3)
    e = GA.entropy(phi, rc, ha, B.F32, ws)
    with torch.autograd.forward_ad.dual_level():
        up = torch.autograd.forward_ad.make_dual(torch.tensor(2.0, dtype=torch.float64),
                                                 torch.tensor(7.0, dtype=torch.float64))
        grad, = torch.autograd.grad(e, phi, grad_outputs=up)
        primal, tangent = torch.autograd.forward_ad.unpack_dual(grad)
    assert torch.equal(primal, 2.0 * column_sums(rc)) and torch.equal(tangent, 7.0 * column_sums(rc))


@pytest.mark.parametrize("factor", [1.0, -2.5])
def test_plain_upstream_gradient(library, factor):
    rc, ha, phi, ws = scene(8)
    grad, = torch.autograd.grad(GA.entropy(phi, rc, ha, B.F32, ws) * factor, phi)
    assert grad.dtype == torch.float32 and torch.equal(grad, factor * column_sums(rc))


def test_upstream_gradient_with_a_pending_negation(library):
    """The imaginary part of a lazily conjugated gradient: its sign is a flag, not in memory."""
    rc, ha, phi, ws = scene(9)
    z = torch.complex(torch.zeros((), dtype=torch.float64), GA.entropy(phi, rc, ha, B.F32, ws))
    loss = (z.conj() * torch.tensor(1 + 2j, dtype=torch.complex128)).real          # 2 E
    grad, = torch.autograd.grad(loss, phi)
    assert torch.equal(grad, 2.0 * column_sums(rc))


@pytest.mark.parametrize("which", ["rc", "ha"])
def test_inference_mode_tensors_are_accepted(library, which):
    rc, ha, phi, ws = scene(4)
    with torch.inference_mode():
        rc, ha = (rc.clone(), ha) if which == "rc" else (rc, ha.clone())
    grad, = torch.autograd.grad(GA.entropy(phi, rc, ha, B.F32, ws), phi)
    assert torch.equal(grad, column_sums(rc))
    assert library.calls == ["entropy", "grad"]   # no version counter to watch: nothing is kept


def test_saved_tensor_hooks_see_the_phase_only(library):
    rc, ha, phi, ws = scene(5)
    seen = []

    def pack(x):
        seen.append(x)
        return x.half()
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda x: x.float()):
        e = GA.entropy(phi, rc, ha, B.F32, ws)
    grad, = torch.autograd.grad(e, phi)
    assert len(seen) == 1 and torch.equal(seen[0], phi.detach())
    assert torch.equal(grad, column_sums(rc)) and library.calls == ["entropy", "grad"]


def test_scene_and_filter_refilled_by_the_library(library, monkeypatch):
    class Refill:
        """Writes its output through the address it gets, as the compiled library does."""

        def __getattr__(self, name):
            def call(*args):
                out = {"sar_range_compress": 2, "bfpfft_exec": 2, "sar_make_filter": 3}[name]
                ctypes.memmove(args[out], new.data_ptr(), new.numel() * 4)
                return B.OK
            return call
    monkeypatch.setattr(B, "_lib", Refill())
    for case in ("range", "exec", "filter"):
        rc, ha, phi, ws = scene(6)
        new = scene(7)[0] if case != "filter" else ha.clone()
        e = GA.entropy(phi, rc, ha, B.F32, ws)
        if case == "range":
            B.sar_range_compress(new, B.F32, rc, B.F32, ha, N_RG, N_AZ, stream=0)
        elif case == "exec":
            B.bfpfft_exec(B.Plan(None, N_AZ, N_RG, B.F32, B.FORWARD), new, rc, stream=0)
        else:
            B.sar_make_filter(new, N_AZ, False, ha, stream=0)
        grad, = torch.autograd.grad(e, phi)
        assert torch.equal(grad, column_sums(rc)), case
        assert library.calls[-1] == "grad", case


def test_only_calls_that_succeed_mark_their_outputs(monkeypatch):
    status = B.OK
    monkeypatch.setattr(B, "_lib", type("Lib", (), {"bfpfft_exec": staticmethod(lambda *a: status),
                                                    "bfpfft_error_string": staticmethod(lambda s: b"")}))
    plan = B.Plan(None, 16, 1, B.F32, B.FORWARD)
    x, y = torch.zeros(16), torch.zeros(16)
    B.bfpfft_exec(plan, x, y, stream=0)
    assert (x._version, y._version) == (0, 1)
    B.bfpfft_exec(plan, x.data_ptr(), y.data_ptr(), stream=0)      # addresses: nothing to mark
    with torch.inference_mode():
        B.bfpfft_exec(plan, x, torch.zeros(16), stream=0)          # no counter to advance
    status = B.ERR_MISALIGNED
    with pytest.raises(B.BfpfftError):
        B.bfpfft_exec(plan, x, y, stream=0)
    assert y._version == 1
