"""The autofocus gradient from a kept image: the same numbers as from one gradient call, at the edges of the range-bin
count, in both storage types; the pass that computes the image again (stream capture) agrees to FP32 rounding; a scene
changed between forward and backward gives the gradient of the changed scene; nothing is kept when no gradient will be
asked for.

The two gradient passes add a CTA's rows in another order, at most 16 rows a CTA here, so they agree to 16 * 2^-24 of
the summands' magnitude; 1e-5 relative L2 leaves room for cancellation between rows.
"""

import pytest

from paper_2605_28451_gb300 import autofocus as GA
from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def scene(n_az, n_rg, dtype, seed=0):
    import torch
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    rc = torch.randn((n_rg, n_az, 2), device="cuda:0", generator=g)
    rc = torch.view_as_complex(rc) if dtype == B.F32 else rc.half()
    ref = torch.from_numpy(synth.centred_reference(synth.azimuth_chirp(128), n_az).astype("complex64")).cuda()
    ha = torch.empty_like(ref)
    B.sar_make_filter(ref, n_az, True, ha)
    phi = torch.from_numpy(synth.phase_error(n_az).astype("float32")).cuda().requires_grad_(True)
    return rc, ha, phi


def direct(rc, dtype, phi, ha, ws):
    import torch
    grad = torch.empty_like(phi)
    B.sar_autofocus_grad(rc, dtype, phi.detach(), ha, rc.shape[1], rc.shape[0], grad, ws.stats, ws.buf, ws.bytes)
    return ws.stats.clone(), grad


@pytest.mark.parametrize("n_az", [256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("n_rg", [1, 3, 37, 1001])
@pytest.mark.parametrize("dtype", [B.F16_BFP, B.F32])
def test_kept_image_gives_the_same_gradient(n_az, n_rg, dtype):
    import torch
    rc, ha, phi = scene(n_az, n_rg, dtype)
    ws = GA.Workspace(n_az, "cuda:0")
    stats, grad = direct(rc, dtype, phi, ha, ws)
    e = GA.entropy(phi, rc, ha, dtype, ws)
    kept, = torch.autograd.grad(e, phi)
    assert torch.equal(e.detach(), stats[2]) and torch.equal(ws.stats, stats)
    assert torch.equal(kept, grad)
    again = torch.empty_like(grad)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):      # inside a capture nothing is kept
        B.sar_autofocus_grad(rc, dtype, phi.detach(), ha, n_az, n_rg, again, ws.stats, ws.buf, ws.bytes)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.linalg.norm(again - grad) <= 1e-5 * torch.linalg.norm(grad)
    assert B.bfpfft_device_status() == B.OK


def test_scene_changed_between_forward_and_backward():
    import torch
    rc, ha, phi = scene(1024, 50, B.F16_BFP)
    ws = GA.Workspace(1024, "cuda:0")
    e = GA.entropy(phi, rc, ha, B.F16_BFP, ws)
    rc.mul_(0.5).add_(0.25)
    got, = torch.autograd.grad(e, phi)
    _, expect = direct(rc, B.F16_BFP, phi, ha, ws)
    assert torch.equal(got, expect)


def test_nothing_is_kept_without_a_gradient(monkeypatch):
    import torch
    rc, ha, phi = scene(4096, 64, B.F16_BFP)
    ws = GA.Workspace(4096, "cuda:0")

    def refuse(*a, **k):
        raise AssertionError("kept an image for an evaluation")
    monkeypatch.setattr(B, "sar_autofocus_entropy_keep", refuse)
    with torch.no_grad():
        GA.entropy(phi, rc, ha, B.F16_BFP, ws)
    GA.entropy(phi.detach(), rc, ha, B.F16_BFP, ws)


def test_bad_states_are_refused():
    import torch
    rc, ha, phi = scene(256, 4, B.F16_BFP)
    ws = GA.Workspace(256, "cuda:0")
    p = phi.detach()
    size = B.sar_autofocus_state_bytes(256, 4)
    host = torch.empty(size, dtype=torch.uint8).pin_memory()
    state = torch.empty(size + 16, dtype=torch.uint8, device="cuda:0")
    for bad, bytes_, status in ((None, size, B.ERR_INVALID_ARG), (host, size, B.ERR_INVALID_ARG),
                                (state, size - 1, B.ERR_INVALID_ARG), (state.data_ptr() + 8, size, B.ERR_MISALIGNED)):
        with pytest.raises(B.BfpfftError) as err:
            B.sar_autofocus_entropy_keep(rc, B.F16_BFP, p, ha, 256, 4, ws.stats, None, bad, bytes_, ws.buf, ws.bytes)
        assert err.value.status == status
    assert B.sar_autofocus_state_bytes(100, 4) == 0


def test_upstream_gradient_scales_the_result():
    import torch
    rc, ha, phi = scene(1024, 20, B.F16_BFP)
    ws = GA.Workspace(1024, "cuda:0")
    _, grad = direct(rc, B.F16_BFP, phi, ha, ws)
    (GA.entropy(phi, rc, ha, B.F16_BFP, ws) * 3.5).backward()
    assert torch.equal(phi.grad, torch.tensor(3.5, device="cuda:0") * grad)
