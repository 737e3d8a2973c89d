"""Particle read-back in the original order: the direct scatter and the
full-sector records (payloads of 64 MiB and more) move bits, so the arrays
returned right after init are the uploaded ones exactly."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,prec,np_", [
    (2, "fp32", (64 << 20) // 20), (2, "fp32", (64 << 20) // 20 + 1), (3, "fp32", (64 << 20) // 28 + 259),
    (2, "fp64", (64 << 20) // 40 + 3), (3, "fp64", (64 << 20) // 56 + 257), (3, "fp32", 1001)])
def test_original_order_bit_exact(torch_cuda, d, prec, np_):
    from paper_2008_09441_gb300 import Run
    torch = torch_cuda
    dt = torch.float32 if prec == "fp32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(np_ + d)
    u = torch.rand(d, np_, generator=g, device="cuda", dtype=dt)
    v = torch.zeros(d, np_, device="cuda", dtype=dt)
    w = torch.rand(np_, generator=g, device="cuda", dtype=dt) - 0.5
    torch.cuda.synchronize()
    run = Run((1.0,) * d, 3, list(u), list(v), w, 0.0, precision=prec)  # dt = 0: nothing moves
    ou, ov, ow = torch.empty_like(u), torch.full_like(v, 7.0), torch.empty_like(w)
    torch.cuda.synchronize()
    run.particles_device(list(ou), list(ov), ow)
    assert torch.equal(ou, u) and torch.equal(ow, w) and not ov.any()
    hu, _, hw = run.particles()
    assert np.array_equal(hu, u.T.cpu().numpy()) and np.array_equal(hw, w.cpu().numpy())
    run.close()
